"""Sequences that the bounded-row engine hands to the engines with backpointer
rows (inputs whose bounds prune little): paths and scores equal those engines'
alone, in batches of like sequences, mixed with ordinary ones, with symbols,
two models, repeated and captured calls."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

GIVEN = 64 + 8 * 64  # byte of the workspace header: sequences handed over, per model


@pytest.fixture(scope="module")
def fv():
    import paper_2510_19301_gb300 as fv
    fv._lib.load(build_if_missing=True)
    return fv


def given(d, m=0):
    return int(np.frombuffer(d.workspace[GIVEN:GIVEN + 256].cpu().numpy().tobytes(), np.int32)[m])


def model(fv, kind, K, g):
    log_pi = torch.log_softmax(torch.randn(K, generator=g, device="cuda"), 0)
    if kind == "equal":
        return fv.Model(torch.zeros(K), torch.full((K, K), -1.0))
    i = torch.arange(K, device="cuda").float()
    A = -0.5 * ((i[:, None] - i[None, :]) / (K / 20)) ** 2
    return fv.Model(log_pi, A - torch.logsumexp(A, 1, keepdim=True))


def scores_of(kind, rows, K, g):
    if kind == "equal":
        return torch.zeros(rows, K, device="cuda")
    return 0.1 * torch.log_softmax(torch.randn(rows, K, generator=g, device="cuda"), -1)


def same(fv, models, b, expect, flags=0):
    d = fv.Decoder(models, b, flags=flags)
    small = fv.Decoder(models, b, workspace=torch.empty(fv.workspace_min_size(models, b), dtype=torch.uint8,
                                                        device="cuda"))
    p, s = (x.clone() for x in small())
    for _ in range(2):
        d.paths.fill_(-1)
        q, r = d()
        assert torch.equal(p, q) and torch.equal(s.view(torch.int32), r.view(torch.int32))
        if expect is not None:
            assert (given(d) > 0) == expect
    return d


@pytest.mark.parametrize("kind", ["flat band", "equal"])
@pytest.mark.parametrize("K,n,T", [(400, 9, 400), (512, 64, 300), (512, 152, 300), (512, 340, 200), (513, 3, 400),
                                   (1000, 30, 300), (1024, 90, 200), (1025, 5, 300), (2048, 9, 200), (2500, 2, 300),
                                   (4096, 8, 150)])
def test_like_sequences(fv, kind, K, n, T):
    g = torch.Generator(device="cuda").manual_seed(K + n)
    m = model(fv, kind, K, g)
    lengths = np.random.default_rng(n).integers(T * 3 // 4, T + 1, n)
    b = fv.Batch(lengths, E=scores_of(kind, int(lengths.sum()), K, g), models=[m])
    # (K = 513: reading every row loses less than 30%; 2048 with nine sequences
    # is near the line)
    same(fv, [m], b, None if K in (513, 2048) else True)


@pytest.mark.parametrize("K,n", [(512, 40), (512, 200), (800, 40), (1400, 12), (4000, 6)])
def test_among_ordinary_sequences(fv, K, n):
    """Scores that order the states of some sequences and not of others."""
    g = torch.Generator(device="cuda").manual_seed(K)
    m = model(fv, "flat band", K, g)
    lengths = np.random.default_rng(K).integers(1, 400, n)
    E = [torch.log_softmax((40.0 if i % 3 else 0.02) * torch.randn(int(t), K, generator=g, device="cuda"), -1)
         for i, t in enumerate(lengths)]
    b = fv.Batch(lengths, E=torch.cat(E), models=[m])
    same(fv, [m], b, None)


def test_symbols_and_two_models(fv):
    rng = np.random.default_rng(3)
    g = torch.Generator(device="cuda").manual_seed(3)
    Ks, V = (520, 1100), 6
    ms = []
    for K in Ks:
        band = model(fv, "flat band", K, g)
        logB = W._log_dirichlet(rng, 50.0, (K, V)).astype(np.float32)
        ms.append(fv.Model(band.log_pi, band.logA, logB=logB))
    idx = np.array([0, 1, 0, 0, 1, 1, 0])
    T = [300, 260, 1, 400, 90, 300, 17]
    obs = rng.integers(0, V, sum(T)).astype(np.int32)
    b = fv.Batch(T, obs=obs, models=ms, model_index=idx)
    d = same(fv, ms, b, None)
    assert given(d, 1) > 0


def test_calls_that_share_the_gpu_keep_large_models(fv):
    g = torch.Generator(device="cuda").manual_seed(1)
    m = model(fv, "equal", 1300, g)
    b = fv.Batch([200, 200], E=scores_of("equal", 400, 1300, g), models=[m])
    same(fv, [m], b, False, flags=fv._lib.FV_SHARED_GPU)


@pytest.mark.parametrize("K", [512, 1000, 1500])
def test_captured(fv, K):
    """One graph, replayed on other scores: handed over, then not."""
    g = torch.Generator(device="cuda").manual_seed(K)
    m = model(fv, "flat band", K, g)
    E = scores_of("flat band", 500, K, g)
    b = fv.Batch([300, 200], E=E, models=[m])
    d = fv.Decoder([m], b)
    d.launch()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        d.launch()
    for sharp in (0, 1, 0):
        E.copy_(torch.log_softmax(60.0 * torch.randn(500, K, generator=g, device="cuda"), -1) if sharp
                else scores_of("flat band", 500, K, g))
        d.paths.fill_(-1)
        graph.replay()
        torch.cuda.synchronize()
        q, r = d.paths.clone(), d.scores.clone()
        assert d.device_status() == 0
        same(fv, [m], b, None)
        ref = fv.Decoder([m], b)()
        assert torch.equal(q, ref[0]) and torch.equal(r, ref[1])
