"""The engines that keep backpointers, which a call reaches through the
smallest workspace (or without host lengths): full-table decoding at every
class of K, symbols included, and dynamic beams, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def fv():
    import paper_2510_19301_gb300 as fv
    fv._lib.load(build_if_missing=True)
    return fv


def bits(a):
    return np.asarray(a, np.float32).view(np.int32)


def check(fv, m, b, lengths, ref, **how):
    ws = torch.empty(fv.workspace_min_size([m], b, **how), dtype=torch.uint8, device="cuda")
    paths, scores = fv.Decoder([m], b, workspace=ws, **how)()
    paths, scores = paths.cpu().numpy(), scores.cpu().numpy()
    o = 0
    for i, (p, s) in enumerate(ref):
        assert np.array_equal(paths[o:o + lengths[i]], p), f"sequence {i} (T={lengths[i]})"
        assert bits(scores[i]) == bits(s)
        o += lengths[i]


@pytest.mark.parametrize("V", [0, 7])
@pytest.mark.parametrize("K", [1, 5, 64, 65, 128, 129, 256, 257, 512, 513, 1000, 1024, 1025, 1500, 2048, 2049])
def test_full_table(fv, K, V):
    rng = np.random.default_rng(K + V)
    log_pi, logA = W.random_model(K, rng)
    if K > 4:
        logA[rng.random((K, K)) < 0.1] = -np.inf
    lengths = [1, 2, 33, 70] if K > 1024 else [1, 2, 33, 90, 150, 7]
    if V:
        logB = W._log_dirichlet(rng, 0.5, (K, V)).astype(np.float32)
        obs = [rng.integers(0, V, t).astype(np.int32) for t in lengths]
        E = [np.ascontiguousarray(logB[:, o].T) for o in obs]
        m = fv.Model(log_pi, logA, logB=logB)
        b = fv.Batch(lengths, obs=np.concatenate(obs), models=[m])
    else:
        E = [W.gaussian_emissions(t, K, rng) for t in lengths]
        m = fv.Model(log_pi, logA)
        b = fv.Batch(lengths, E=torch.from_numpy(np.concatenate(E)).cuda(), models=[m])
    hmm = oracle.HMM(log_pi, logA)
    check(fv, m, b, lengths, oracle.map_sequences(lambda e: oracle.viterbi(hmm, e), E))


@pytest.mark.parametrize("K,B,n", [(200, 30, 5), (300, 64, 170), (600, 200, 5), (1024, 100, 5), (1300, 90, 3)])
def test_dynamic_beam(fv, K, B, n):
    rng = np.random.default_rng(K)
    log_pi, logA = W.random_model(K, rng)
    lengths = [int(t) for t in rng.integers(1, 40, n)]
    E = [W.gaussian_emissions(t, K, rng) for t in lengths]
    m = fv.Model(log_pi, logA)
    b = fv.Batch(lengths, E=torch.from_numpy(np.concatenate(E)).cuda(), models=[m])
    hmm = oracle.HMM(log_pi, logA)
    check(fv, m, b, lengths, oracle.map_sequences(lambda e: oracle.beam(hmm, e, B)[:2], E), mode="beam", B=B, P=0)
