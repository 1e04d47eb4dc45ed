"""Top-B select of the one-block beam kernel (FLASH-BS; dynamic beams of small
CSR models): thresholds that move or jump from step to step, bins with more
equal scores than are ranked, signed zeros, against the oracle bit for bit."""
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


@pytest.mark.parametrize("form", ["dense_bs", "csr_bs", "csr_dyn"])
@pytest.mark.parametrize("B", [33, 128])
@pytest.mark.parametrize("kind", ["plain", "ties", "scale", "jump", "negzero"])
def test_beam_select(fv, kind, B, form):
    K = 515
    rng = np.random.default_rng(B)
    log_pi, logA = W.random_model(K, rng)
    rp, col, val = W.random_csr(K, 40, rng)
    T = [1, 2, 40, 75]
    E = [W.gaussian_emissions(t, K, rng) for t in T]
    if kind == "ties":
        logA = rng.integers(-2, 3, logA.shape).astype(np.float32)
        val = rng.integers(-2, 3, val.shape).astype(np.float32)
        log_pi = rng.integers(-2, 3, K).astype(np.float32)
        E = [rng.integers(-1, 2, e.shape).astype(np.float32) for e in E]
    elif kind == "negzero":
        logA = np.where(rng.random(logA.shape) < 0.5, -0.0, 0.0).astype(np.float32)
        val = np.where(rng.random(val.shape) < 0.5, -0.0, 0.0).astype(np.float32)
        log_pi = np.where(rng.random(K) < 0.5, -0.0, 0.0).astype(np.float32)
        E = [np.where(rng.random(e.shape) < 0.5, -0.0, -1.0).astype(np.float32) for e in E]
    elif kind == "scale":
        E = [(e * np.where(np.arange(len(e)) % 7 == 3, 1e4, 1e-3)[:, None]).astype(np.float32) for e in E]
    elif kind == "jump":
        E = [(e + np.where(np.arange(len(e)) % 5 == 2, 3e3, -8e2)[:, None]).astype(np.float32) for e in E]
    if form == "dense_bs":
        m, hmm = fv.Model(log_pi, logA), oracle.HMM(log_pi, logA)
    else:
        m, hmm = fv.Model(log_pi, row_ptr=rp, col=col, val=val), oracle.HMM(log_pi, None, rp, col, val)
    P = 0 if form == "csr_dyn" else 3
    b = fv.Batch(T, E=torch.from_numpy(np.concatenate(E)).cuda(), models=[m])
    paths, scores = fv.decode([m], b, mode="beam", B=B, P=P)
    paths, scores = paths.cpu().numpy(), scores.cpu().numpy()
    run = (lambda e: oracle.flash_bs(hmm, e, P, B)) if P else (lambda e: oracle.beam(hmm, e, B))
    o = 0
    for i, r in enumerate(oracle.map_sequences(run, E)):
        assert r[-1] == 0
        assert np.array_equal(paths[o:o + T[i]], r[0]), f"{kind} B={B} sequence {i}"
        assert np.float32(scores[i]).view(np.int32) == np.float32(r[1]).view(np.int32)
        o += T[i]
