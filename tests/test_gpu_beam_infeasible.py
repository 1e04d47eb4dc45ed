"""A dynamic beam that empties is reported; the scores of the call's other
sequences are written all the same, also where one CTA or cluster decodes
several sequences in turn."""
import numpy as np
import pytest

import oracle
import workloads as W

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("K,n,shared", [(150, 500, 0), (300, 400, 0), (600, 250, 0), (600, 400, 1), (1030, 100, 0)])
def test_other_sequences_keep_their_scores(K, n, shared):
    import paper_2510_19301_gb300 as fv
    fv._lib.load(build_if_missing=True)
    rng = np.random.default_rng(K)
    log_pi, logA = W.random_model(K, rng)
    B, T = 20, 6
    E = [W.gaussian_emissions(T, K, rng) for _ in range(n)]
    dead = [i for i in range(n) if i % 17 == 0]
    for k, i in enumerate(dead):
        E[i][k % T] = -np.inf
    m = fv.Model(log_pi, logA)
    b = fv.Batch([T] * n, E=torch.from_numpy(np.concatenate(E)).cuda(), models=[m])
    d = fv.Decoder([m], b, mode="beam", B=B, P=0, flags=fv._lib.FV_SHARED_GPU if shared else 0)
    d.scores.fill_(float("nan"))
    d.launch()
    assert d.device_status() == fv._lib.FV_EINFEASIBLE
    scores = d.scores.cpu().numpy()
    hmm = oracle.HMM(log_pi, logA)
    live = [i for i in range(n) if i not in set(dead)]
    ref = oracle.map_sequences(lambda i: oracle.beam(hmm, E[i], B)[1], live)
    assert np.array_equal(scores[live].view(np.int32), np.asarray(ref, np.float32).view(np.int32))
