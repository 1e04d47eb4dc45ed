"""Top-B select of the CSR cluster beam (K >= 8192, B >= 64): thresholds that
move from step to step, bins with more equal scores than are ranked, beams
wider than the candidates, against the oracle bit for bit."""
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


@pytest.mark.parametrize("B", [64, 200, 3000])
@pytest.mark.parametrize("kind", ["plain", "ties", "scale", "jump", "negzero"])
def test_csr_cluster_select(fv, kind, B):
    K, deg = 8200, 9
    rng = np.random.default_rng(B)
    rp, col, val = W.random_csr(K, deg, rng)
    log_pi = W._log_dirichlet(rng, 1.0, (K,)).astype(np.float32)
    T = [1, 2, 12, 30]
    E = [W.gaussian_emissions(t, K, rng) for t in T]
    if kind == "ties":
        val = rng.integers(-2, 3, val.shape).astype(np.float32)
        log_pi = rng.integers(-2, 3, K).astype(np.float32)
        E = [rng.integers(-1, 2, e.shape).astype(np.float32) for e in E]
    elif kind == "negzero":
        val = np.where(rng.random(val.shape) < 0.5, -0.0, 0.0).astype(np.float32)
        log_pi = np.where(rng.random(K) < 0.5, -0.0, 0.0).astype(np.float32)
        E = [np.where(rng.random(e.shape) < 0.5, -0.0, -1.0).astype(np.float32) for e in E]
    elif kind == "scale":
        E = [(e * np.where(np.arange(len(e)) % 7 == 3, 1e4, 1e-3)[:, None]).astype(np.float32) for e in E]
    elif kind == "jump":
        E = [(e + np.where(np.arange(len(e)) % 5 == 2, 3e3, -8e2)[:, None]).astype(np.float32) for e in E]
    m = fv.Model(log_pi, row_ptr=rp, col=col, val=val)
    hmm = oracle.HMM(log_pi, None, rp, col, val)
    b = fv.Batch(T, E=torch.from_numpy(np.concatenate(E)).cuda(), models=[m])
    paths, scores = fv.decode([m], b, mode="beam", B=B, P=0)
    paths, scores = paths.cpu().numpy(), scores.cpu().numpy()
    o = 0
    for i, r in enumerate(oracle.map_sequences(lambda e: oracle.beam(hmm, e, B), E)):
        assert r[-1] == 0
        assert np.array_equal(paths[o:o + T[i]], r[0]), f"{kind} B={B} sequence {i}"
        assert np.float32(scores[i]).view(np.int32) == np.float32(r[1]).view(np.int32)
        o += T[i]
