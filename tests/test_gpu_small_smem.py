"""Shared memory of the K <= 128 engines: a staged symbol table with direct
FLASH rows behind it, around the 48 KB that a launch may use without asking.
The sizes run upwards in a fresh process, where no larger call has raised the
limit before; every result against the oracle."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

pytest.importorskip("torch")

# (K, V, T, P): the longest segment of T / P states keeps T / P - 1 rows of 64
# or 128 bytes behind a table of V such rows of floats
CASES = [
    (128, 64, 2000, 16),  # 32768 + 15872 bytes
    (128, 53, 2576, 16), (128, 55, 2576, 16), (128, 56, 2576, 16), (100, 54, 2576, 16),  # + 20480
    (64, 149, 2576, 16), (64, 151, 2576, 16), (64, 152, 2576, 16), (40, 150, 2576, 16),  # + 10240
    (128, 92, 3000, 2), (128, 96, 3000, 2), (64, 188, 3000, 2), (64, 192, 3000, 2),  # the table alone
    (128, 97, 700, 4), (64, 193, 700, 4),  # not staged
]

SCRIPT = """
import numpy as np, torch
import oracle, workloads as W
import paper_2510_19301_gb300 as fv
fv._lib.load(build_if_missing=True)
bad = []
for K, V, T, P in %r:
    rng = np.random.default_rng(K + V)
    log_pi, logA = W.random_model(K, rng)
    logB = W._log_dirichlet(rng, 0.5, (K, V)).astype(np.float32)
    obs = rng.integers(0, V, T).astype(np.int32)
    p, s = oracle.viterbi(oracle.HMM(log_pi, logA), np.ascontiguousarray(logB[:, obs].T))
    m = fv.Model(log_pi, logA, logB=logB)
    b = fv.Batch([T], obs=obs, models=[m])
    small = torch.empty(fv.workspace_min_size([m], b), dtype=torch.uint8, device="cuda")
    for how in (dict(mode="flash", P=P), dict(mode="flash", P=P, flags=fv._lib.FV_COMPLETE_PRUNING),
                dict(mode="checkpoint", P=0), dict(workspace=small), dict()):
        try:
            q, r = fv.Decoder([m], b, **how)()
            ok = np.array_equal(q.cpu().numpy(), p) if "flags" not in how else True
            ok = ok and np.float32(r[0].item()).view(np.int32) == np.float32(s).view(np.int32)
        except fv.FVError as e:
            ok = False
        if not ok:
            how.pop("workspace", None)
            bad.append((K, V, T, P, how))
print("BAD", bad)
"""


def test_tables_and_rows_around_48_kb():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", SCRIPT % (CASES,)], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    assert r.stdout.strip().endswith("BAD []"), r.stdout[-2000:]
