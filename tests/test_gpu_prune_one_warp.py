"""The configurations of the bounded-row engine whose jobs have one warp per
CTA (K <= 256 in large batches, 256 < K <= 512 up to 120 sequences): the
lanes of that warp hand each other every step's delta through shared memory.
All paths and scores against the engines with backpointer rows."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("K,n,T", [(131, 900, 120), (256, 2000, 200), (257, 17, 300), (512, 120, 250)])
def test_every_sequence_equals_the_backpointer_engines(K, n, T):
    import paper_2510_19301_gb300 as fv
    fv._lib.load(build_if_missing=True)
    rng = np.random.default_rng(K + n)
    log_pi, logA = W.random_model(K, rng)
    lengths = rng.integers(T * 9 // 10, T + 1, n)
    m = fv.Model(log_pi, logA)
    g = torch.Generator(device="cuda").manual_seed(K)
    E = torch.log_softmax(torch.randn(int(lengths.sum()), K, generator=g, device="cuda"), dim=-1)
    b = fv.Batch(lengths, E=E, models=[m])
    dec = fv.Decoder([m], b)
    small = fv.Decoder([m], b, workspace=torch.empty(fv.workspace_min_size([m], b), dtype=torch.uint8, device="cuda"))
    p, s = (x.clone() for x in small())
    for _ in range(3):
        dec.paths.fill_(-1)
        q, r = dec()
        assert torch.equal(p, q) and torch.equal(s.view(torch.int32), r.view(torch.int32))
