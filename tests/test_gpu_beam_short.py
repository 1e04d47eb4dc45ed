"""Dynamic beams on either side of the lengths from which the bounded-row engine
takes them (8, 32 and 48 steps by K and call), against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("K,B,T", [(511, 30, [3, 7]), (512, 100, [31, 4]), (512, 100, [32, 4]), (600, 50, [7, 1]),
                                   (600, 50, [8]), (1024, 64, [47]), (1024, 64, [48, 2]), (1100, 90, [7]),
                                   (1100, 90, [8, 3])])
@pytest.mark.parametrize("shared", [0, 1])
def test_short_beams(K, B, T, shared):
    import paper_2510_19301_gb300 as fv
    fv._lib.load(build_if_missing=True)
    rng = np.random.default_rng(K + T[0])
    log_pi, logA = W.random_model(K, rng)
    E = [W.gaussian_emissions(t, K, rng) for t in T]
    m = fv.Model(log_pi, logA)
    b = fv.Batch(T, E=torch.from_numpy(np.concatenate(E)).cuda(), models=[m])
    paths, scores = fv.decode([m], b, mode="beam", B=B, P=0, flags=fv._lib.FV_SHARED_GPU if shared else 0)
    paths, scores = paths.cpu().numpy(), scores.cpu().numpy()
    hmm = oracle.HMM(log_pi, logA)
    o = 0
    for i, e in enumerate(E):
        p, s = oracle.beam(hmm, e, B)[:2]
        assert np.array_equal(paths[o:o + T[i]], p)
        assert np.float32(scores[i]).view(np.int32) == np.float32(s).view(np.int32)
        o += T[i]
