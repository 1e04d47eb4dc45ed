"""FLASH at K <= 128: the first level whose tasks fit the direct rows (160) is
solved in one launch.  Segments of 159 .. 162 rows on either side of the line,
levels above it, ragged batches; paths and scores equal exact decoding's."""
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


@pytest.mark.parametrize("K,V", [(1, 0), (5, 3), (64, 0), (65, 40), (128, 0)])
@pytest.mark.parametrize("P,lengths", [(2, [320, 321, 322, 323, 324, 325]), (1, [2, 3, 160, 161, 162]),
                                       (4, [5, 640, 647, 1300, 30]), (16, [40, 16, 17, 5200])])
def test_direct_levels(fv, K, V, P, lengths):
    rng = np.random.default_rng(K + P)
    log_pi, logA = W.random_model(K, rng)
    if K > 4:
        logA[rng.random((K, K)) < 0.2] = -np.inf
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
    paths, scores = fv.decode([m], b, mode="flash", P=P)
    paths, scores = paths.cpu().numpy(), scores.cpu().numpy()
    hmm = oracle.HMM(log_pi, logA)
    o = 0
    for i, (p, s) in enumerate(oracle.map_sequences(lambda e: oracle.viterbi(hmm, e), E)):
        assert np.array_equal(paths[o:o + lengths[i]], p), f"K={K} P={P} sequence {i} (T={lengths[i]})"
        assert np.float32(scores[i]).view(np.int32) == np.float32(s).view(np.int32)
        o += lengths[i]
