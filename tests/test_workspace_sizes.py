"""The two workspace sizes of a request, and the Decoder's step down to the
smaller one when the device cannot hold the larger.  Needs no GPU: sizes are
computed on the host, and the allocation is a stand-in that refuses."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def fv():
    import paper_2510_19301_gb300 as fv
    fv._lib.load(build_if_missing=True)
    return fv


def request_of(fv, K, T):
    log_pi, logA = W.random_model(K, np.random.default_rng(K))
    m = fv.Model(log_pi, logA, device="cpu")
    return m, fv.Batch(T, E=torch.empty(1), models=[m], device="cpu")


def table(K, T, size):
    """Bytes of a table of `size`-byte entries, each sequence's rounded up to
    eight entries."""
    return sum((t * K + 7) // 8 * 8 for t in T) * size


@pytest.mark.parametrize("K", [5, 64, 128, 200, 512, 1000, 1500, 4096])
def test_smallest_size_is_the_backpointer_table(fv, K):
    T = [400, 3, 91]
    m, b = request_of(fv, K, T)
    small, big = fv.workspace_min_size([m], b), fv.workspace_size([m], b)
    assert table(K, T, 2) < small <= big and big > table(K, T, 4)
    # a hundred sequences more add the two tables, and under 4 KB each besides
    m2, b2 = m, fv.Batch(T + [50] * 100, E=torch.empty(1), models=[m], device="cpu")
    assert fv.workspace_min_size([m2], b2) - small < table(K, [50] * 100, 2) + 100 * 4096


@pytest.mark.parametrize("mode,kw", [("flash", dict(P=4)), ("checkpoint", dict(P=0)), ("flash", dict(P=4, mem_budget=1 << 16))])
def test_other_modes_have_one_size(fv, mode, kw):
    m, b = request_of(fv, 200, [300, 40])
    assert fv.workspace_min_size([m], b, mode=mode, **kw) == fv.workspace_size([m], b, mode=mode, **kw)


def test_table_beyond_half_of_the_memory(fv):
    """35e9 state-steps: 140 GB of delta rows next to 140 GB of emission
    scores.  From there the request asks for 2-byte backpointers."""
    K = 512
    m, b = request_of(fv, K, [300_000] * 260)
    total = 260 * 300_000 * K
    assert fv.workspace_size([m], b) == fv.workspace_min_size([m], b) < 2.1 * total
    m, b = request_of(fv, K, [300_000] * 30)
    assert fv.workspace_size([m], b) > 4 * 30 * 300_000 * K


@pytest.mark.parametrize("mode,B", [("vanilla", 0), ("beam", 16)])
def test_decoder_steps_down_when_memory_is_short(fv, monkeypatch, mode, B):
    K, T = 300, [7000, 20]
    m, b = request_of(fv, K, T)
    kw = dict(mode=mode, B=B, P=0) if mode == "beam" else dict(mode=mode)
    big, small = fv.workspace_size([m], b, **kw), fv.workspace_min_size([m], b, **kw)
    assert small < big
    empty = torch.empty

    def limited(n, *a, limit=big, **k):
        if k.get("dtype") is not torch.uint8:
            return empty(n, *a, **k)
        if n >= limit:
            raise torch.cuda.OutOfMemoryError("no room")
        x = empty(n + 256, *a, **k)
        o = -x.data_ptr() % 256
        return x[o:o + n]

    monkeypatch.setattr(torch, "empty", limited)
    d = fv.Decoder([m], b, **kw)
    assert d.ws_bytes == small == d.workspace.numel()
    monkeypatch.setattr(torch, "empty", lambda n, *a, **k: limited(n, *a, limit=small, **k))
    with pytest.raises(torch.cuda.OutOfMemoryError):
        fv.Decoder([m], b, **kw)
