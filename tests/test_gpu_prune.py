"""The bounded-row engine (exact decoding, 128 < K <= 4096): paths and scores
against the oracle, bit for bit, at the edges of its tiles, launch
configurations and trace segments, and on inputs that bound badly."""
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


def check(fv, log_pi, logA, E_list, pad=0, sample=None):
    """Decode E_list packed from element `pad` of the emission buffer; compare
    the sampled sequences (all by default) with the oracle."""
    K = log_pi.shape[0]
    T = [e.shape[0] for e in E_list]
    flat = np.concatenate([np.zeros(pad, np.float32)] + [e.reshape(-1) for e in E_list])
    off = pad + np.concatenate([[0], np.cumsum(np.asarray(T, np.int64) * K)[:-1]])
    m = fv.Model(log_pi, logA)
    b = fv.Batch(T, E=torch.from_numpy(flat).cuda(), models=[m], e_off=off)
    paths, scores = fv.decode([m], b)
    paths, scores = paths.cpu().numpy(), scores.cpu().numpy()
    hmm = oracle.HMM(log_pi, logA)
    pick = range(len(T)) if sample is None else sample
    ref = oracle.map_sequences(lambda i: oracle.viterbi(hmm, E_list[i]), list(pick))
    start = np.concatenate([[0], np.cumsum(T)])
    for i, (p, s) in zip(pick, ref):
        assert np.array_equal(paths[start[i]:start[i] + T[i]], p), f"K={K} sequence {i} (T={T[i]}) path"
        assert bits(scores[i]) == bits(s), f"K={K} sequence {i} score"


# tile edges of every padded size; segments of the trace are 48 states here,
# their warm-up 24
@pytest.mark.parametrize("K", [129, 130, 131, 255, 256, 257, 383, 511, 512, 513, 897, 1023, 1024])
def test_tile_and_segment_edges(fv, K):
    rng = np.random.default_rng(K)
    log_pi, logA = W.random_model(K, rng)
    T = [1, 2, 3, 47, 48, 49, 71, 72, 73, 74, 96, 97, 121, 145]
    check(fv, log_pi, logA, [W.gaussian_emissions(t, K, rng) for t in T], pad=K % 3)


@pytest.mark.parametrize("K,T", [(1025, [1, 49, 73, 90]), (1500, [2, 50, 97]), (2048, [48, 75]), (2049, [1, 51, 74]),
                                 (3000, [60]), (4095, [49]), (4096, [50, 2])])
def test_large_state_spaces(fv, K, T):
    rng = np.random.default_rng(K)
    log_pi, logA = W.random_model(K, rng, alpha=0.1 if K % 2 else 1.0)
    check(fv, log_pi, logA, [W.gaussian_emissions(t, K, rng) for t in T], pad=K % 3)


# launch configurations: jobs per SM and steps against the longest sequence
@pytest.mark.parametrize("K,n,T", [(256, 1300, 40), (200, 700, 33), (300, 119, 30), (300, 121, 30), (512, 160, 25),
                                   (512, 400, 20), (700, 170, 20)])
def test_launch_configurations(fv, K, n, T):
    rng = np.random.default_rng(n)
    log_pi, logA = W.random_model(K, rng)
    lengths = rng.integers(max(1, T - 5), T + 1, n)
    E = [W.gaussian_emissions(int(t), K, rng) for t in lengths]
    check(fv, log_pi, logA, E, sample=sorted(rng.choice(n, 24, replace=False)))


@pytest.mark.parametrize("K", [144, 300, 600, 1100])
@pytest.mark.parametrize("kind", ["flat", "spikes", "ties", "sparse", "constant", "negzero", "wide"])
def test_inputs_that_bound_badly(fv, K, kind):
    rng = np.random.default_rng(K)
    log_pi, logA = W.random_model(K, rng)
    T = [60, 1, 75, 130]
    E = [W.gaussian_emissions(t, K, rng) for t in T]
    if kind == "flat":  # emissions that order no state
        E = [(1e-3 * e).astype(np.float32) for e in E]
    elif kind == "spikes":  # one huge weight per column, and columns without any
        logA[rng.integers(0, K, K), np.arange(K)] = 40.0
        logA[:, rng.integers(0, K, 5)] = -np.inf
    elif kind == "ties":
        logA = rng.integers(-3, 4, (K, K)).astype(np.float32)
        log_pi = rng.integers(-3, 4, K).astype(np.float32)
        E = [rng.integers(-3, 4, e.shape).astype(np.float32) for e in E]
    elif kind == "sparse":  # few finite edges: whole columns inside their lists
        logA[rng.random((K, K)) < 0.985] = -np.inf
        log_pi[rng.random(K) < 0.9] = -np.inf
    elif kind == "constant":  # every candidate equal at every step
        logA[:] = -1.0
        log_pi[:] = 0.0
        E = [np.zeros_like(e) for e in E]
    elif kind == "negzero":  # zeros of both signs meet in the maximum
        logA = np.where(rng.random((K, K)) < 0.5, -0.0, 0.0).astype(np.float32)
        log_pi = np.where(rng.random(K) < 0.5, -0.0, 0.0).astype(np.float32)
        E = [np.where(rng.random(e.shape) < 0.9, -0.0, 0.0).astype(np.float32) for e in E]
    elif kind == "wide":  # magnitudes where a margin must cover the roundings
        logA = (1e4 * rng.standard_normal((K, K))).astype(np.float32)
        E = [(1e6 * rng.standard_normal(e.shape)).astype(np.float32) for e in E]
    check(fv, log_pi, logA, E)


def test_wrong_segment_ends_are_traced_again(fv):
    """Two disconnected halves whose scores cross at the last step: the best
    state of every earlier step lies off the path, so every segment is
    re-traced to its start."""
    K, T = 160, 400
    rng = np.random.default_rng(5)
    log_pi, logA = W.random_model(K, rng)
    h = K // 2
    logA[:h, h:] = -np.inf
    logA[h:, :h] = -np.inf
    E = W.gaussian_emissions(T, K, rng)
    E[0, h:] += 50.0
    E[T - 1, :h] += 100.0
    check(fv, log_pi, logA, [E])


def test_symbols_and_two_models(fv):
    rng = np.random.default_rng(8)
    Ks, V = [150, 260], 11
    prm = [W.random_model(K, rng) + (W._log_dirichlet(rng, 0.5, (K, V)).astype(np.float32),) for K in Ks]
    idx = np.array([0, 1, 1, 0, 0, 1])
    T = [50, 1, 120, 49, 7, 96]
    obs = [rng.integers(0, V, t).astype(np.int32) for t in T]
    ms = [fv.Model(a, b, logB=c) for a, b, c in prm]
    b = fv.Batch(T, obs=np.concatenate(obs), models=ms, model_index=idx)
    paths, scores = fv.decode(ms, b)
    paths, scores = paths.cpu().numpy(), scores.cpu().numpy()
    o = 0
    for i, t in enumerate(T):
        lp, lA, lB = prm[idx[i]]
        p, s = oracle.viterbi(oracle.HMM(lp, lA), np.ascontiguousarray(lB[:, obs[i]].T))
        assert np.array_equal(paths[o:o + t], p) and bits(scores[i]) == bits(s)
        o += t


@pytest.mark.parametrize("K", [256, 512])
def test_small_workspace_keeps_the_backpointer_engines(fv, K):
    """A workspace of the backpointer table's size (smaller than the delta
    rows) decodes with the other engines to the same result."""
    rng = np.random.default_rng(3)
    log_pi, logA = W.random_model(K, rng)
    T = [6000, 700, 33]
    m = fv.Model(log_pi, logA)
    b = fv.Batch(T, E=torch.from_numpy(W.gaussian_emissions(sum(T), K, rng)).cuda(), models=[m])
    big = fv.Decoder([m], b)
    ws = torch.empty(big.ws_bytes * 3 // 4, dtype=torch.uint8, device="cuda")
    small = fv.Decoder([m], b, workspace=ws)
    p0, s0 = (x.clone() for x in big())
    p1, s1 = small()
    assert torch.equal(p0, p1) and torch.equal(s0, s1)


def check_beam(fv, log_pi, logA, E_list, B, flags=0):
    K = log_pi.shape[0]
    T = [e.shape[0] for e in E_list]
    m = fv.Model(log_pi, logA)
    b = fv.Batch(T, E=torch.from_numpy(np.concatenate(E_list)).cuda(), models=[m])
    paths, scores = fv.decode([m], b, mode="beam", B=B, P=0, flags=flags)
    paths, scores = paths.cpu().numpy(), scores.cpu().numpy()
    hmm = oracle.HMM(log_pi, logA)
    o = 0
    for i, r in enumerate(oracle.map_sequences(lambda e: oracle.beam(hmm, e, B), E_list)):
        assert r[-1] == 0
        assert np.array_equal(paths[o:o + T[i]], r[0]), f"K={K} B={B} sequence {i} (T={T[i]}) path"
        assert bits(scores[i]) == bits(r[1]), f"K={K} B={B} sequence {i} score"
        o += T[i]


# every padded size, one and several CTAs per sequence (the shared-GPU flag
# keeps one at K <= 1024); 80 sequences: one CTA each
@pytest.mark.parametrize("K,B,n,shared", [(129, 7, 4, 0), (256, 255, 4, 0), (257, 64, 4, 1), (512, 100, 4, 0), (513, 33, 4, 0),
                                          (1024, 256, 4, 0), (1000, 200, 4, 1), (700, 90, 80, 0), (1025, 128, 3, 0),
                                          (2048, 500, 2, 0)])
def test_beam_sizes(fv, K, B, n, shared):
    rng = np.random.default_rng(K + B)
    log_pi, logA = W.random_model(K, rng)
    T = [1, 2, 49, 80][:n] if n <= 4 else list(rng.integers(1, 30, n))
    check_beam(fv, log_pi, logA, [W.gaussian_emissions(int(t), K, rng) for t in T], B,
               flags=fv._lib.FV_SHARED_GPU if shared else 0)


# the select: one bin holds more candidates than are ranked (equal scores,
# one common value, scores of another scale from step to step), B = 1, B >= K
@pytest.mark.parametrize("K", [150, 600, 1100])
@pytest.mark.parametrize("kind,B", [("ties", 40), ("equal", 100), ("scale", 64), ("plain", 1), ("plain", 5000),
                                    ("jump", 90)])
def test_beam_select(fv, K, kind, B):
    rng = np.random.default_rng(K + B)
    log_pi, logA = W.random_model(K, rng)
    T = [40, 1, 60]
    E = [W.gaussian_emissions(t, K, rng) for t in T]
    if kind == "ties":
        logA = rng.integers(-2, 3, (K, K)).astype(np.float32)
        log_pi = rng.integers(-2, 3, K).astype(np.float32)
        E = [rng.integers(-1, 2, e.shape).astype(np.float32) for e in E]
    elif kind == "equal":
        logA[:] = -2.0
        log_pi[:] = -0.0
        E = [np.zeros_like(e) for e in E]
    elif kind == "scale":
        E = [(e * np.where(np.arange(len(e)) % 7 == 3, 1e4, 1e-3)[:, None]).astype(np.float32) for e in E]
    elif kind == "jump":  # the common level of the scores moves by far more than their spread
        E = [(e + np.where(np.arange(len(e)) % 5 == 2, 3e3, -8e2)[:, None]).astype(np.float32) for e in E]
    check_beam(fv, log_pi, logA, E, B)


@pytest.mark.parametrize("K", [200, 900])
def test_beam_that_empties_is_reported(fv, K):
    rng = np.random.default_rng(K)
    log_pi, logA = W.random_model(K, rng)
    logA[:, :] = -np.inf
    m = fv.Model(log_pi, logA)
    b = fv.Batch([20, 5], E=torch.from_numpy(W.gaussian_emissions(25, K, rng)).cuda(), models=[m])
    d = fv.Decoder([m], b, mode="beam", B=16, P=0)
    d.launch()
    assert d.device_status() == fv._lib.FV_EINFEASIBLE
