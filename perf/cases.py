"""The decoding work that users of this framework run, as measurable cases.

A case is a dict of plain values.  ``kind`` says which public entry point a
pass goes through:

* ``exact``  -- Decoder(mode = vanilla / flash / checkpoint), one launch;
* ``decode`` -- the one-call ``decode()``: structs, workspace and outputs made
  on the call and the device status read back, as a script calls it;
* ``beam``   -- Decoder(mode = beam) on dense transitions (P = 0: dynamic
  beam, P >= 1: FLASH-BS);
* ``csr``    -- Decoder(mode = beam) on a sparse random graph;
* ``train``  -- emission layer, ViterbiScore, backward: one training step's
  gradients.

Inputs are synthetic HMMs of the families the benchmark and the tests use:
Dirichlet rows (dense), Erdos-Renyi graphs with absent edges and sampled
symbols, Gaussian log-softmax emission scores, a 32-successor sparse graph,
and CRF-style unnormalised transition scores.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2510_19301_gb300 as fv

DEV = "cuda"


def listed():
    return [
        # a script that tags a handful of short sentences with a small tag set
        # (an odd K) through the one-call API: latency and host work
        dict(name="tag_k37_onecall", kind="decode", K=37, n=5, tlo=3, thi=40, spread="uniform", model="crf", V=0,
             mode="vanilla", P=1, budget=0, shared=False),
        # one symbol sequence of a 64-state HMM: the plain single-request decode
        dict(name="one_k64_symbols", kind="exact", K=64, n=1, tlo=1000, thi=1000, spread="uniform", model="dirichlet",
             alpha=1.0, V=32, mode="vanilla", P=1, budget=0, shared=False),
        # the paper's synthetic default point (Erdos-Renyi, K = T = 512, 50
        # symbols, p = 0.253), one request
        dict(name="er_k512_one", kind="exact", K=512, n=1, tlo=512, thi=512, spread="uniform", model="er", p=0.253,
             V=50, mode="vanilla", P=1, budget=0, shared=False),
        # one launch of the serving loop: 70 exact requests of the 64-state
        # class, lengths log-uniform over the serving range
        dict(name="serve_k64_exact", kind="exact", K=64, n=70, tlo=100, thi=20000, spread="log", model="dirichlet",
             alpha=1.0, V=0, mode="vanilla", P=1, budget=0, shared=True),
        # the headline batch: 1024 sequences of uneven length, K = 256, full
        # backpointers
        dict(name="batch_k256_vanilla", kind="exact", K=256, n=1024, tlo=500, thi=4000, spread="uniform",
             model="dirichlet", alpha=1.0, V=0, mode="vanilla", P=1, budget=0, shared=False),
        # FLASH divide and conquer under 1/16 of the backpointer table, on a
        # batch that leaves part of the chip's slots empty
        dict(name="batch_k256_flash_budget", kind="exact", K=256, n=301, tlo=500, thi=4000, spread="uniform",
             model="dirichlet", alpha=1.0, V=0, mode="flash", P=16, budget=16, shared=False),
        # a batch over a state space that no tile divides
        dict(name="batch_k1000_vanilla", kind="exact", K=1000, n=150, tlo=200, thi=1500, spread="uniform",
             model="dirichlet", alpha=1.0, V=0, mode="vanilla", P=1, budget=0, shared=False),
        # large state space, peaked (Dirichlet 0.1) rows, a batch of 8 long
        # sequences: the whole GPU on one lockstep batch
        dict(name="long_k4096_vanilla", kind="exact", K=4096, n=8, tlo=1500, thi=1500, spread="uniform",
             model="dirichlet", alpha=0.1, V=0, mode="vanilla", P=1, budget=0, shared=False),
        # structured-perceptron / CRF training step: 512 sentences, 128 tags,
        # a 256-feature emission layer, gradients of every parameter
        dict(name="train_k128_crf", kind="train", K=128, n=512, tlo=20, thi=512, spread="uniform", D=256, P=16),
        # one launch of the serving loop's beam class at K = 1024
        dict(name="serve_k1024_beam", kind="beam", K=1024, n=40, tlo=100, thi=2000, spread="log", model="dirichlet",
             alpha=1.0, V=0, B=256, P=0, shared=True),
        # the paper's FLASH-BS on its synthetic default point
        dict(name="er_k512_flash_bs", kind="beam", K=512, n=1, tlo=512, thi=512, spread="uniform", model="er",
             p=0.253, V=50, B=128, P=16, shared=False),
        # sparse 65536-state decoding graph, batch of 8, wide beam
        dict(name="sparse_k65536_beam", kind="csr", K=65536, n=8, tlo=600, thi=600, spread="uniform", deg=32, B=512),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the listed families with sizes over their whole ranges.  The
    cells of an exact pass (sum T K^2), the cells of a beam pass (sum T B K)
    and the emission scores (sum T K) are bounded by the listed cases'."""
    fam = rng.choice(["exact", "exact", "exact", "exact", "decode", "beam", "csr", "train"])
    if fam == "train":
        return dict(kind="train", K=_log_int(rng, 8, 160), n=_log_int(rng, 8, 512), tlo=20,
                    thi=_log_int(rng, 40, 512), spread="uniform", D=rng.choice([64, 100, 256]), P=rng.choice([4, 16]))
    if fam == "csr":
        K = _log_int(rng, 8192, 65536)
        return dict(kind="csr", K=K, n=rng.randint(1, 8), tlo=50, thi=_log_int(rng, 100, 600), spread="uniform",
                    deg=rng.choice([8, 16, 32]), B=_log_int(rng, 64, 1024))
    model = rng.choice(["dirichlet", "dirichlet", "er", "crf"])
    V = rng.choice([32, 50]) if model == "er" else rng.choice([0, 0, 32])
    c = dict(kind=fam, model=model, V=V, spread=rng.choice(["uniform", "log"]), shared=False)
    if model == "dirichlet":
        c["alpha"] = rng.choice([1.0, 1.0, 0.1])
    if model == "er":
        c["p"] = rng.choice([0.1, 0.253, 0.6])
    if fam == "decode":
        c.update(K=_log_int(rng, 4, 300), n=rng.randint(1, 8), tlo=rng.randint(1, 8), thi=rng.randint(10, 60),
                 mode=rng.choice(["vanilla", "flash"]), P=4, budget=0)
    elif fam == "beam":
        K = _log_int(rng, 32, 2048)
        c.update(K=K, B=max(4, K // rng.choice([2, 4, 8, 16])), P=rng.choice([0, 0, 4]), shared=rng.random() < 0.5)
        n = _log_int(rng, 1, 64)
        top = max(64, min(2000, int(6e9 / (n * K * c["B"]))))
        c.update(n=n, tlo=max(8, top // 20), thi=top)
    else:
        K = _log_int(rng, 24, 4096)
        n = _log_int(rng, 1, 8 if K > 1024 else 256)
        top = max(64, min(8000, int(4e10 / (n * K * K)), int(2e8 / (n * K))))
        mode = rng.choice(["vanilla", "vanilla", "vanilla", "flash", "flash", "checkpoint"])
        c.update(K=K, n=n, tlo=max(2, top // rng.choice([1, 4, 50])), thi=top, mode=mode,
                 P=0 if mode == "checkpoint" else rng.choice([4, 16]), budget=16 if mode == "flash" else 0)
    return c


# ---------------------------------------------------------------- inputs
def _lengths(case):
    """The lengths belong to the case (its outputs keep their shapes); the
    seed draws the models, the scores and the symbols."""
    lo, hi, n = case["tlo"], case["thi"], case["n"]
    r = np.random.default_rng([lo, hi, n, case["K"]])
    if case["spread"] == "log":
        return np.floor(np.exp(r.uniform(math.log(lo), math.log(hi + 1), n))).astype(np.int32).clip(lo, hi)
    return r.integers(lo, hi + 1, n).astype(np.int32)


def _log_gamma_draws(alpha, shape, g):
    """log of Gamma(alpha) draws in float64; small alpha through
    Gamma(alpha) = Gamma(alpha + 1) U^(1/alpha), which does not underflow."""
    if alpha >= 1.0:
        return torch._standard_gamma(torch.full(shape, alpha, dtype=torch.float64, device=DEV), generator=g).log()
    x = torch._standard_gamma(torch.full(shape, alpha + 1.0, dtype=torch.float64, device=DEV), generator=g).log()
    u = torch.rand(shape, generator=g, dtype=torch.float64, device=DEV).clamp_min(1e-300)
    return x + u.log() / alpha


def _log_dirichlet(alpha, shape, g):
    x = _log_gamma_draws(alpha, shape, g)
    return (x - torch.logsumexp(x, dim=-1, keepdim=True)).float()


def _dense_model(case, g):
    """(log_pi [K], logA [K, K]) float32 on the device."""
    K = case["K"]
    if case["model"] == "crf":
        return (0.5 * torch.randn(K, generator=g, device=DEV), 0.5 * torch.randn(K, K, generator=g, device=DEV))
    log_pi = _log_dirichlet(1.0, (K,), g)
    if case["model"] == "er":
        x = _log_gamma_draws(1.0, (K, K), g)
        keep = torch.rand(K, K, generator=g, device=DEV) < case["p"]
        one = torch.randint(K, (K, 1), generator=g, device=DEV)
        keep.scatter_(1, one, True)  # every state keeps an out-edge
        x = torch.where(keep, x, torch.full_like(x, -math.inf))
        return log_pi, (x - torch.logsumexp(x, dim=-1, keepdim=True)).float()
    return log_pi, _log_dirichlet(case["alpha"], (K, K), g)


def _symbols(log_pi, logA, logB, lengths, g):
    """Symbols sampled from the HMM itself, all sequences side by side."""
    n, tmax = len(lengths), int(lengths.max())
    gum = lambda lp: lp - torch.empty_like(lp).exponential_(generator=g).log()  # noqa: E731
    A, B = logA.double(), logB.double()
    q = gum(log_pi.double().expand(n, -1).contiguous()).argmax(1)
    out = torch.empty(n, tmax, dtype=torch.int32, device=DEV)
    for t in range(tmax):
        if t:
            q = gum(A[q]).argmax(1)
        out[:, t] = gum(B[q]).argmax(1)
    rows = torch.arange(tmax, device=DEV)[None, :] < torch.as_tensor(lengths, device=DEV)[:, None]
    return out[rows]


def _emissions(rows, K, g):
    E = torch.empty(rows, K, device=DEV)
    for r in range(0, rows, 1 << 19):
        x = torch.randn(min(rows - r, 1 << 19), K, generator=g, device=DEV)
        E[r:r + x.shape[0]] = torch.log_softmax(x, dim=-1)
    return E


def _csr(case, g):
    """deg distinct sorted successors per state, log Dirichlet(1) weights."""
    K, deg = case["K"], case["deg"]
    col = torch.randint(K - deg, (K, deg), generator=g, device=DEV).sort(dim=1).values
    col = (col + torch.arange(deg, device=DEV)).int()
    val = _log_dirichlet(1.0, (K, deg), g)
    ptr = torch.arange(K + 1, device=DEV, dtype=torch.int32) * deg
    return _log_dirichlet(1.0, (K,), g), ptr, col, val


def _inputs(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    T = _lengths(case)
    rows = int(T.sum())
    if case["kind"] == "csr":
        return T, _csr(case, g), _emissions(rows, case["K"], g)
    if case["kind"] == "train":
        K, D = case["K"], case["D"]
        return T, dict(log_pi=0.5 * torch.randn(K, generator=g, device=DEV),
                       logA=0.5 * torch.randn(K, K, generator=g, device=DEV),
                       W=torch.randn(K, D, generator=g, device=DEV) / 16.0,
                       b=torch.randn(K, generator=g, device=DEV) / 16.0), torch.randn(rows, D, generator=g, device=DEV)
    log_pi, logA = _dense_model(case, g)
    if case["V"]:
        logB = _log_dirichlet(0.5 if case["model"] != "er" else 1.0, (case["K"], case["V"]), g)
        return T, (log_pi, logA, logB), _symbols(log_pi, logA, logB, T, g)
    return T, (log_pi, logA, None), _emissions(rows, case["K"], g)


def _flags(case):
    return fv._lib.FV_SHARED_GPU if case.get("shared") else 0


def _how(case, T):
    if case["kind"] == "csr":
        return dict(mode="beam", B=case["B"], P=0)
    if case["kind"] == "beam":
        return dict(mode="beam", B=case["B"], P=case["P"], flags=_flags(case))
    how = dict(mode=case["mode"], P=case["P"], flags=_flags(case))
    if case["budget"]:
        how["mem_budget"] = int(T.astype(np.int64).sum()) * case["K"] * 2 // case["budget"]
    return how


def prepare(case, seed):
    T, params, data = _inputs(case, seed)
    if case["kind"] == "train":
        for p in params.values():
            p.requires_grad_(True)
        return dict(kind="train", lengths=T, X=data, P=case["P"], **params)
    if case["kind"] == "csr":
        log_pi, ptr, col, val = params
        m = fv.Model(log_pi, row_ptr=ptr, col=col.reshape(-1), val=val.reshape(-1))
    else:
        m = fv.Model(params[0], params[1], logB=params[2])
    if m.logB is not None:
        b = fv.Batch(T, obs=data, models=[m])
    else:
        b = fv.Batch(T, E=data, models=[m])
    if case["kind"] == "decode":
        return dict(kind="decode", model=m, batch=b, how=_how(case, T))
    return dict(kind="decoder", decoder=fv.Decoder([m], b, **_how(case, T)))


def run(state):
    if state["kind"] == "decoder":
        return state["decoder"](check=False)
    if state["kind"] == "decode":
        return fv.decode(state["model"], state["batch"], **state["how"])
    W, bias, log_pi, logA = state["W"], state["b"], state["log_pi"], state["logA"]
    E = torch.addmm(bias, state["X"], W.t())
    scores = fv.ViterbiScore.apply(log_pi, logA, E, state["lengths"], "flash", state["P"])
    grads = torch.autograd.grad(scores.sum(), (log_pi, logA, W, bias))
    return [scores.detach(), *grads]


def work(case):
    """Inputs read once, paths and scores (or gradients) written once; two
    operations (add, max) per candidate of the recursion."""
    T = _lengths(case).astype(np.float64)
    K, n, steps = case["K"], case["n"], float(T.sum())
    out = 4.0 * steps + 4.0 * n
    if case["kind"] == "csr":
        # of E only the entries of states that the beam reaches are needed
        reach = min(K, case["B"] * case["deg"])
        return dict(bytes=4.0 * steps * reach + 8.0 * K * case["deg"] + out, flops=2.0 * steps * reach)
    if case["kind"] == "train":
        D = case["D"]
        return dict(bytes=4.0 * (steps * D + 2 * K * (K + D + 2)) + 4.0 * n,
                    flops=2.0 * steps * K * K + 4.0 * steps * K * D)
    src = case["B"] if case["kind"] == "beam" else K
    emit = 4.0 * steps if case["V"] else 4.0 * steps * K
    return dict(bytes=emit + 4.0 * K * (K + 1 + case["V"]) + out, flops=2.0 * steps * src * K)


# ---------------------------------------------------------------- 64 bits
class _Emit:
    """Emission scores of step t of sequences [0, a), in float64, the
    sequences sorted by falling length."""

    def __init__(self, T, data, logB):
        self.order = np.argsort(-T, kind="stable")
        off = np.concatenate([[0], np.cumsum(T.astype(np.int64))])[:-1][self.order]
        self.T, self.off = T[self.order], torch.as_tensor(off, device=DEV)
        self.data, self.logB = data, None if logB is None else logB.double()

    def active(self, t):
        return int((self.T > t).sum())

    def __call__(self, t, a):
        x = self.data[self.off[:a] + t]
        return x.double() if self.logB is None else self.logB[:, x.long()].t()

    def unsort(self, x):
        out = torch.empty_like(x)
        out[torch.as_tensor(self.order, device=DEV)] = x
        return out


def _exact_scores(T, log_pi, logA, logB, data, B=None, back=False):
    """Best path score of every sequence (within the beam of the B best
    states per step, if B is given), in float64; back: the paths too."""
    em = _Emit(T, data, logB)
    AT = logA.double().t().contiguous()  # [target, source]
    K, n = AT.shape[0], len(T)
    score = torch.empty(n, dtype=torch.float64, device=DEV)
    psi, last = [], torch.empty(n, dtype=torch.int64, device=DEV)
    d = log_pi.double() + em(0, n)
    chunk = max(1, int(1.5e9 / (8 * K * K)))
    for t in range(int(T.max())):
        a = em.active(t)
        if t:
            best = torch.empty(a, K, dtype=torch.float64, device=DEV)
            arg = torch.empty(a, K, dtype=torch.int64, device=DEV) if back else None
            for s in range(0, a, chunk):
                c = d[s:min(a, s + chunk), None, :] + AT
                if back:
                    best[s:s + chunk], arg[s:s + chunk] = c.max(2)
                else:
                    best[s:s + chunk] = c.amax(2)
            d = best + em(t, a)
            if back:
                psi.append(arg)
        if B is not None and B < K:
            v = d.topk(B, dim=1).values[:, -1:]
            d = torch.where(d >= v, d, torch.full_like(d, -math.inf))
        done = em.active(t + 1)
        score[done:a], last[done:a] = d[done:].max(1)
        d = d[:done]
    if not back:
        return em.unsort(score)
    paths = torch.zeros(n, int(T.max()), dtype=torch.int64, device=DEV)
    q = last
    for t in range(int(T.max()) - 1, -1, -1):
        a = em.active(t)
        paths[:a, t] = q[:a]
        if t:
            q[:a] = psi[t - 1].gather(1, q[:a, None])[:, 0]
    return em.unsort(score), em.unsort(paths)


def _exact_csr(T, params, data, B):
    log_pi, _, col, val = params
    em = _Emit(T, data, None)
    n, K, deg = len(T), log_pi.shape[0], col.shape[1]
    col, val = col.long(), val.double()
    score = torch.empty(n, dtype=torch.float64, device=DEV)
    d = log_pi.double() + em(0, n)
    for t in range(int(T.max())):
        a = em.active(t)
        if t:
            v, i = d.topk(min(B, K), dim=1)
            c = v[:a, :, None] + val[i[:a]]
            d = torch.full((a, K), -math.inf, dtype=torch.float64, device=DEV)
            d.scatter_reduce_(1, col[i[:a]].reshape(a, -1), c.reshape(a, -1), "amax")
            d += em(t, a)
        done = em.active(t + 1)
        score[done:a] = d[done:].max(1).values
        d = d[:done]
    return em.unsort(score)


def exact(case, seed):
    T, params, data = _inputs(case, seed)
    if case["kind"] == "csr":
        return [None, _exact_csr(T, params, data, case["B"])]
    if case["kind"] == "beam":
        if case["P"]:  # the score is of the path that the segment beams leave
            return None
        return [None, _exact_scores(T, *params, data, B=case["B"])]
    if case["kind"] != "train":
        return [None, _exact_scores(T, *params, data)]
    K, W, X = case["K"], params["W"].double(), data.double()
    E = X @ W.t() + params["b"].double()
    scores, paths = _exact_scores(T, params["log_pi"], params["logA"], None, E, back=True)
    rows = torch.arange(paths.shape[1], device=DEV)[None, :] < torch.as_tensor(T, device=DEV)[:, None]
    dpi = torch.bincount(paths[:, 0], minlength=K).double()
    pairs = (paths[:, :-1] * K + paths[:, 1:])[rows[:, 1:]]
    dA = torch.bincount(pairs, minlength=K * K).double().reshape(K, K)
    dE = torch.nn.functional.one_hot(paths[rows], K).double()
    return [scores, dpi, dA, dE.t() @ X, dE.sum(0)]
