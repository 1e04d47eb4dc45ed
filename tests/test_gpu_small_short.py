"""Exact decoding at K <= 128 on either side of the lengths from which values
only are kept (40, 112 and 144 steps by K and number of sequences), with
sequences of every length beside the longest, against the oracle."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("longest", [1, 39, 40, 49, 111, 112, 143, 144, 200])
@pytest.mark.parametrize("K,V,n", [(1, 0, 9), (8, 0, 9), (37, 5, 9), (64, 0, 9), (64, 0, 320), (100, 0, 9), (128, 7, 9),
                                   (128, 0, 170)])
def test_lengths(K, V, n, longest):
    import paper_2510_19301_gb300 as fv
    fv._lib.load(build_if_missing=True)
    rng = np.random.default_rng(K + longest)
    log_pi, logA = W.random_model(K, rng)
    if K > 4:
        logA[rng.random((K, K)) < 0.2] = -np.inf
    T = [longest] + [min(longest, t) for t in (1, 2, 47, 48, 49, 73, 97, 121)]
    T += [int(t) for t in rng.integers(1, longest + 1, n - len(T))]
    if V:
        logB = W._log_dirichlet(rng, 0.5, (K, V)).astype(np.float32)
        obs = [rng.integers(0, V, t).astype(np.int32) for t in T]
        E = [np.ascontiguousarray(logB[:, o].T) for o in obs]
        m = fv.Model(log_pi, logA, logB=logB)
        b = fv.Batch(T, obs=np.concatenate(obs), models=[m])
    else:
        E = [W.gaussian_emissions(t, K, rng) for t in T]
        m = fv.Model(log_pi, logA)
        b = fv.Batch(T, E=torch.from_numpy(np.concatenate(E)).cuda(), models=[m])
    paths, scores = fv.decode([m], b)
    paths, scores = paths.cpu().numpy(), scores.cpu().numpy()
    hmm = oracle.HMM(log_pi, logA)
    o = np.concatenate([[0], np.cumsum(T)])
    pick = list(range(min(n, 24)))
    for i, (p, s) in zip(pick, oracle.map_sequences(lambda i: oracle.viterbi(hmm, E[i]), pick)):
        assert np.array_equal(paths[o[i]:o[i + 1]], p), f"sequence {i} (T={T[i]})"
        assert np.float32(scores[i]).view(np.int32) == np.float32(s).view(np.int32)
