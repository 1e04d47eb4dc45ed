"""Dynamic beams spread over a four-CTA cluster (1024 < K <= 2048): every CTA
sends its columns of a step by bulk copies and masks them at the start of the
next step.  Narrow beams mask nearly every column; all sequences against the
decoding that keeps a sequence on one CTA."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("K,B", [(1025, 3), (1400, 60), (2048, 8), (2048, 700)])
def test_cluster_beams_equal_one_cta_beams(K, B):
    import paper_2510_19301_gb300 as fv
    fv._lib.load(build_if_missing=True)
    rng = np.random.default_rng(K + B)
    log_pi, logA = W.random_model(K, rng)
    lengths = rng.integers(150, 201, 24)
    m = fv.Model(log_pi, logA)
    g = torch.Generator(device="cuda").manual_seed(K)
    E = torch.log_softmax(torch.randn(int(lengths.sum()), K, generator=g, device="cuda"), dim=-1)
    b = fv.Batch(lengths, E=E, models=[m])
    one = fv.Decoder([m], b, mode="beam", B=B, P=0, flags=fv._lib.FV_SHARED_GPU)
    many = fv.Decoder([m], b, mode="beam", B=B, P=0)
    p, s = one()
    for _ in range(3):
        many.paths.fill_(-1)
        q, r = many()
        assert torch.equal(p, q) and torch.equal(s.view(torch.int32), r.view(torch.int32))
