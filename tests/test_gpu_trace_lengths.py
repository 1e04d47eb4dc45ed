"""The lengths on the device are the ones decoded.  Where they differ from the
host's copy (used for planning) and the workspace holds them, every state of
every path is still written: the trace's launch is sized from the host's
lengths."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("K,mode,host,device", [
    (64, "vanilla", [20], [400]), (64, "vanilla", [100, 3], [700, 260]), (200, "vanilla", [48], [49]),
    (200, "vanilla", [60, 40], [500, 1]), (600, "vanilla", [30], [300]), (1100, "vanilla", [10, 10], [150, 60]),
    (300, "beam", [200, 200], [385, 10]), (300, "beam", [30, 30, 30], [80, 5, 3]),
])
def test_device_lengths_beyond_the_hosts(K, mode, host, device):
    import paper_2510_19301_gb300 as fv
    fv._lib.load(build_if_missing=True)
    rng = np.random.default_rng(K + sum(device))
    log_pi, logA = W.random_model(K, rng)
    E = [W.gaussian_emissions(t, K, rng) for t in device]
    m = fv.Model(log_pi, logA)
    b = fv.Batch(device, E=torch.from_numpy(np.concatenate(E)).cuda(), models=[m])
    how = dict(mode=mode, B=40, P=0) if mode == "beam" else dict(mode=mode)
    ws = torch.empty(fv.workspace_size([m], b, **how) + (1 << 20), dtype=torch.uint8, device="cuda")
    b.T_host = np.asarray(host, np.int32)
    d = fv.Decoder([m], b, workspace=ws, **how)
    d.paths.fill_(-1)
    paths, scores = d()
    paths, scores = paths.cpu().numpy(), scores.cpu().numpy()
    hmm = oracle.HMM(log_pi, logA)
    o = 0
    for i, e in enumerate(E):
        p, s = (oracle.beam(hmm, e, 40) if mode == "beam" else oracle.viterbi(hmm, e))[:2]
        assert np.array_equal(paths[o:o + device[i]], p), f"sequence {i}"
        assert np.float32(scores[i]).view(np.int32) == np.float32(s).view(np.int32)
        o += device[i]
