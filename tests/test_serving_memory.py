"""The serving loop's memory accounting: a request counts with the table its
launch really keeps, and one that fits the budget only with 2-byte
backpointers is served in that workspace.  Runs on the host: tensors on the
CPU, a stand-in for the prepared decoder."""
import pytest

torch = pytest.importorskip("torch")

import paper_2510_19301_gb300 as fv  # noqa: E402
from paper_2510_19301_gb300.serve import GpuBackend, Request, Server  # noqa: E402


class RecordedDecoder:
    def __init__(self, models, batch, workspace=None, **how):
        self.models, self.batch, self.how = models, batch, how
        self.ws_bytes = fv.workspace_size(models, batch, **how) if workspace is None else workspace.numel()


class HostBackend(GpuBackend):
    def __init__(self):
        fv._lib.load(build_if_missing=True)
        self.torch, self.Batch, self.Model, self.Decoder = torch, fv.Batch, fv.Model, RecordedDecoder
        self.workspace_min_size = fv.workspace_min_size
        self.FV_SHARED_GPU = fv._lib.FV_SHARED_GPU
        self.device, self.shared, self.model_seed, self._models = "cpu", True, 6, {}
        self.launched = []

    def launch_batch(self, reqs):
        dec, E, _ = self._batch_decoder(reqs)
        small = dec.ws_bytes == fv.workspace_min_size(dec.models, dec.batch, **dec.how)
        self.launched.append((sorted(r.rid for r in reqs), dec.ws_bytes, 4 * E.numel(), small))
        return {"n": len(reqs)}

    def poll(self, h):
        return 0

    def result(self, h, i=0):
        return None

    def release(self, h):
        pass


@pytest.mark.parametrize("K,T", [(64, 2000), (256, 900), (1000, 2500)])
def test_budget_covers_what_the_launch_holds(K, T):
    be = HostBackend()
    reqs = [Request(rid=i, K=K, T=T) for i in range(8)]
    need = be.bytes_needed(reqs[0])
    srv = Server(be, mem_budget_bytes=3 * need, clock=iter(x * 1e-3 for x in range(10 ** 6)).__next__)
    rep = srv.run(reqs, realtime=False)
    assert rep["requests"] == 8 and rep["failed"] == 0
    # beyond the rows, a launch keeps copies of the model (two of K x 1024 at
    # most here) and tables of a few bytes per step
    model = 2 * 4 * K * 1024 + (1 << 18)
    assert all(len(r) <= 3 and ws + e <= 3 * need + model for r, ws, e, _ in be.launched)


def test_request_that_fits_only_with_backpointers_is_served():
    K, T = 200, 4000
    be = HostBackend()
    big, other = Request(rid=0, K=K, T=T), Request(rid=1, K=K, T=T // 4)
    full = be.bytes_needed(big)
    budget = full - T * K  # 4 bytes per state-step do not fit, 2 do
    srv = Server(be, mem_budget_bytes=budget, clock=iter(x * 1e-3 for x in range(10 ** 6)).__next__)
    rep = srv.run([big, other, Request(rid=2, K=K, T=2 * T)], realtime=False)
    assert rep["requests"] == 2 and [r.rid for r in srv.failed] == [2] and srv.peak_bytes <= budget
    compact = {tuple(r): c for r, _, _, c in be.launched}
    assert compact == {(0,): True, (1,): False}
