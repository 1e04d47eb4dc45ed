"""A variant tuned for one kind of decoding stays with it: tuning FLASH or
Checkpoint leaves full-table decoding on its own engine, and tuning full-table
decoding finds a variant for the others without leaving that engine unless
a variant beats it."""
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


def request_of(fv, K, n, T):
    rng = np.random.default_rng(K)
    log_pi, logA = W.random_model(K, rng)
    E = [W.gaussian_emissions(T, K, rng) for _ in range(n)]
    m = fv.Model(log_pi, logA)
    return m, fv.Batch([T] * n, E=torch.from_numpy(np.concatenate(E)).cuda(), models=[m]), (log_pi, logA, E)


@pytest.mark.parametrize("K", [64, 256, 400, 1000])
@pytest.mark.parametrize("mode,kw", [("flash", dict(P=4)), ("checkpoint", dict(P=0))])
def test_other_modes_leave_full_tables_alone(fv, K, mode, kw):
    m, b, _ = request_of(fv, K, 6, 120)
    try:
        chosen = fv.autotune([m], b, mode=mode, **kw)
        assert fv.engine_variant(K, "flash") == fv.engine_variant(K, "checkpoint") == chosen[0]
        assert fv.engine_variant(K, "vanilla") == 0
    finally:
        fv.set_engine_variant(K, 0)


@pytest.mark.parametrize("K", [64, 256, 400, 1000])
def test_full_tables_keep_the_faster_engine(fv, K):
    m, b, (log_pi, logA, E) = request_of(fv, K, 40, 400)
    n = fv.set_engine_variant(K, 0)
    try:
        chosen = fv.autotune([m], b)
        assert fv.engine_variant(K, "vanilla") == chosen[0]
        assert 0 <= fv.engine_variant(K, "flash") < n
        paths, scores = fv.decode([m], b)
        p, s = oracle.viterbi(oracle.HMM(log_pi, logA), E[0])
        assert np.array_equal(paths[:400].cpu().numpy(), p)
        assert np.float32(scores[0].item()).view(np.int32) == np.float32(s).view(np.int32)
        fv.set_engine_variant(K, n - 1)
        assert fv.engine_variant(K, "vanilla") == fv.engine_variant(K, "flash") == n - 1
    finally:
        fv.set_engine_variant(K, 0)
