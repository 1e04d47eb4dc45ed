#!/usr/bin/env python3
"""Benchmark of the FLASH Viterbi decoding hot path on one GB300.

Workload (default): 1024 sequences, K = 256 dense FP32 log-transitions
(Dirichlet(1) rows), per-step emission scores log_softmax(N(0,1)), T uniform
in [500, 4000]; one batched, uneven-length decode per step.  The metric is
state-steps/s = sum_b T_b * K per second.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--mode vanilla|flash]
    python bench.py --impl reference      # the CPU oracle on the host cores

Under torchrun (N > 1) every rank decodes its own batch (weak scaling, no
collective on the data path); rank 0 prints one JSON line.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "state-steps/s (sum T*K) vs plain GPU Viterbi, bit-exact paths; serving p99 latency"
UNIT = "state-steps/s"
WORKLOAD = "batched-uneven: 1024 seqs, K=256 dense FP32, T~U[500,4000], E=log_softmax(N(0,1))"


# DRAM bytes per state-step of prune_fwd_kernel (K=256, vanilla, the default
# engine): reads of E plus writes of the delta rows, from one ncu capture
# (dram__bytes_read.sum + dram__bytes_write.sum) of a 608-sequence launch of
# 1000 steps.
DRAM_BYTES_PER_STATE_STEP = (622936576 + 573162496) / (608 * 1000 * 256)
TRAFFIC_VARIANT = 0  # the configuration those counters were taken on


def dist_env():
    return int(os.environ.get("RANK", 0)), int(os.environ.get("WORLD_SIZE", 1)), int(os.environ.get("LOCAL_RANK", 0))


def rank_seed(rank):
    """Each rank decodes its own batch (weak scaling): same shape, its own
    seeded lengths and emission scores."""
    return 2 + 7919 * rank


def aggregate_ranks(ms, units, device="cpu"):
    """Whole-job throughput over the ranks of the process group (if any):
    the units all ranks processed divided by the slowest rank's time.
    Returns (value per second, max ms, total units)."""
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(ms)], dtype=torch.float64, device=device)
    u = torch.tensor([float(units)], dtype=torch.float64, device=device)
    if dist.is_available() and dist.is_initialized() and dist.get_world_size() > 1:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        dist.all_reduce(u, op=dist.ReduceOp.SUM)
    ms_max, total = float(t.item()), float(u.item())
    return total / (ms_max / 1e3), ms_max, total


class ClockSampler:
    """nvidia-smi samples every 200 ms during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.gpu = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), "--query-gpu=" + self.Q, "--format=csv,noheader,nounits",
                 "-lms", "200"], stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None
        time.sleep(0.3)

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"], "samples": 0}
        time.sleep(0.25)
        self.proc.terminate()
        self.proc.wait()
        rows = []
        for line in open(self.path):
            f = [x.strip() for x in line.split(",")]
            if len(f) >= 9:
                rows.append(f)
        os.unlink(self.path)
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        reasons = set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            for k, n in enumerate(names):
                if r[5 + k].lower().startswith("active"):
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(rows)}


def peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return d, "measured"
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "sm_max_mhz": 2070.0}, "fallback"


def sm_count(device=None):
    import torch
    return int(torch.cuda.get_device_properties(device or torch.cuda.current_device()).multi_processor_count)


def alu_peak_tops(sm_mhz, sms=None):
    """FP32 CUDA-core max-plus peak: SMs x 128 FP32 lanes x 2 ops x clock,
    i.e. one cell (one add + one max) per lane per cycle, the analogue of
    counting an FFMA as 2 flops."""
    return (sms or sm_count()) * 128 * 2 * sm_mhz * 1e6 / 1e12


def measured_alu_peak(fv, iters=200000):
    """The library's register-only max-plus probe (fv_maxplus_peak): the
    decode engines' add.f32x2 + 3-input max pair on every SM, CUDA events."""
    cps, per_clk, sms = fv.maxplus_peak(iters)
    return {"tflops": 2.0 * cps / 1e12, "cells_per_clk_per_sm": per_clk, "sm_count": sms}


def make_workload(args, rank, device):
    import torch

    import paper_2510_19301_gb300 as fv
    import workloads as W
    K = args.K
    log_pi, logA = W.config2_model(seed=2, K=K)
    lengths = W.config2_lengths(seed=rank_seed(rank), n_seq=args.n_seq)
    E = W.gaussian_emissions_packed_device(int(lengths.sum()), K, seed=rank_seed(rank), device=device)
    m = fv.Model(log_pi, logA, device=device)
    return dict(K=K, log_pi=log_pi, logA=logA, lengths=lengths, E=E, model=m)


def cpu_baseline(wl, seconds_target=20.0):
    """The oracle as it stands, on the host cores, one sequence per thread,
    over a bounded sample of the same batch (first sequences in batch order)."""
    import oracle
    oracle.build()
    K = wl["K"]
    lengths = wl["lengths"]
    hmm = oracle.HMM(wl["log_pi"], wl["logA"])
    cores = os.cpu_count() or 1
    n = min(len(lengths), 8 * cores)
    e_off = np.concatenate([[0], np.cumsum(lengths.astype(np.int64) * K)])
    Eflat = wl["E"].view(-1)
    jobs = [Eflat[e_off[i]:e_off[i + 1]].view(-1, K).cpu().numpy() for i in range(n)]
    t0 = time.perf_counter()
    oracle.map_sequences(lambda e: oracle.viterbi(hmm, e), jobs, threads=cores)
    dt = time.perf_counter() - t0
    steps = int(lengths[:n].astype(np.int64).sum()) * K
    return {"value": steps / dt, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"first {n} of {len(lengths)} sequences ({steps} state-steps), exact vanilla oracle, "
                      f"{cores} threads, {dt:.2f} s wall"}


def time_decoder(dec, steps, warmup, lib):
    """Device time per step (CUDA events on the launching stream) and the
    mean duration of the library's main decode kernels per step."""
    import ctypes

    import torch
    for _ in range(warmup):
        dec.launch()
    torch.cuda.synchronize()
    st = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    lib.fv_timing_enable(1)
    e0.record(st)
    for _ in range(steps):
        dec.launch()
    e1.record(st)
    torch.cuda.synchronize()
    tot, npairs = ctypes.c_float(0), ctypes.c_int32(0)
    lib.fv_timing_read(ctypes.byref(tot), ctypes.byref(npairs))
    lib.fv_timing_enable(0)
    return e0.elapsed_time(e1) / steps, tot.value / max(steps, 1)


def flash_phases(dec, lib):
    """One FLASH decode with the library's timing pairs: the root pass (with
    its resolve), then every task level of Alg. 1 (a budget decode's last
    level is its leaf waves).  Returns the milliseconds per phase."""
    import ctypes

    import torch
    torch.cuda.synchronize()
    lib.fv_timing_enable(1)
    dec.launch()
    buf = (ctypes.c_float * 256)()
    n = ctypes.c_int32(0)
    lib.fv_timing_pairs(buf, 256, ctypes.byref(n))
    lib.fv_timing_enable(0)
    ms = [float(buf[i]) for i in range(n.value)]
    return {"root_pass_ms": ms[0] if ms else None, "task_level_ms": ms[1:],
            "levels": max(0, len(ms) - 1)}


def per_sequence_comparator(fv, m, lengths, E, K, n_sample, device):
    """Plain GPU Viterbi: the same exact decoder launched once per sequence
    (one sequence per call, one stream), timed on a sample of sequences."""
    import torch
    e_off = np.concatenate([[0], np.cumsum(lengths.astype(np.int64) * K)])
    decs = []
    for i in range(n_sample):
        Ei = E.view(-1)[e_off[i]:e_off[i + 1]]
        decs.append(fv.Decoder([m], fv.Batch([int(lengths[i])], E=Ei, models=[m], device=device)))
    for d in decs:
        d.launch()
    torch.cuda.synchronize()
    st = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(st)
    for d in decs:
        d.launch()
    e1.record(st)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    steps = int(lengths[:n_sample].astype(np.int64).sum()) * K
    return {"value": steps / (ms / 1e3), "unit": UNIT, "sample": f"first {n_sample} sequences, one launch each",
            "ms": ms}


def config1_latency(fv, device, iters=200):
    """One K=64 sequence of T=1000 discrete symbols (the small, latency-bound
    workload): device time per decode, as back-to-back fv_decode calls and
    as a CUDA graph replay of one decode."""
    import torch

    import workloads as W
    w = W.config1()
    m = fv.Model(w["log_pi"], w["logA"], logB=w["logB"], device=device)
    b = fv.Batch([w["T"]], obs=w["obs"], models=[m], device=device)
    steps = w["T"] * w["K"]
    st = torch.cuda.Stream(device=device)
    out = {"workload": "1 sequence, K=64, V=32 symbols, T=1000 (discrete emissions)"}
    ref = None
    for name, kw in (("vanilla", {"mode": "vanilla"}), ("flash_P16", {"mode": "flash", "P": 16}),
                     ("beam_B16", {"mode": "beam", "B": 16, "P": 0})):
        if name == "vanilla":
            # engine configuration picked for this one-sequence request
            out["engine_variant"] = int(fv.autotune([m], b, mode="vanilla")[0])
        d = fv.Decoder([m], b, **kw)
        with torch.cuda.stream(st):
            d(st, check=True)
            for _ in range(5):
                d.launch(st)
        st.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        for _ in range(iters):
            d.launch(st)
        e1.record(st)
        st.synchronize()
        us_launch = e0.elapsed_time(e1) * 1e3 / iters
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=st):
            d.launch(st)
        for _ in range(3):
            g.replay()
        torch.cuda.synchronize()
        e0.record(st)
        with torch.cuda.stream(st):
            for _ in range(iters):
                g.replay()
        e1.record(st)
        st.synchronize()
        us_graph = e0.elapsed_time(e1) * 1e3 / iters
        assert d.device_status(st) == 0
        row = {"us_per_decode": us_launch, "us_per_decode_graph": us_graph,
               "value": steps / (us_graph / 1e6), "unit": UNIT}
        if name == "vanilla":
            ref = (d.paths.clone(), d.scores.clone())
        elif name == "flash_P16":
            row["bit_identical_to_vanilla"] = bool(torch.equal(ref[0], d.paths) and torch.equal(
                ref[1].view(torch.int32), d.scores.view(torch.int32)))
        out[name] = row
        del g, d
    return out


def config4_train(fv, device, steps=10, warmup=3):
    """One training step of the CRF-style tagger (K=128 tags, 512 sequences
    of 20..512 steps, 256 features): E = X W^T + b (a plain FP32 library
    GEMM, TF32 off), scores = ViterbiScore (FLASH P=16 decode), loss = sum
    of scores, backward (path counts through the emission layer)."""
    import torch

    import workloads as W
    w = W.config4()
    prev_tf32 = torch.backends.cuda.matmul.allow_tf32
    torch.backends.cuda.matmul.allow_tf32 = False
    try:
        X = torch.from_numpy(w["X"]).to(device)
        Wt = torch.from_numpy(w["W"]).to(device).requires_grad_(True)
        bias = torch.from_numpy(w["b"]).to(device).requires_grad_(True)
        log_pi = torch.from_numpy(w["log_pi"]).to(device).requires_grad_(True)
        logA = torch.from_numpy(w["logA"]).to(device).requires_grad_(True)
        lengths = w["T"]

        # engine configuration of the K=128 class picked on this batch
        with torch.no_grad():
            E0 = X @ Wt.t() + bias
        m0 = fv.Model(log_pi.detach(), logA.detach(), device=device)
        tuned = int(fv.autotune([m0], fv.Batch(lengths, E=E0.reshape(-1), models=[m0], device=device),
                                mode="flash", P=16)[0])
        del E0

        def step():
            for p in (Wt, bias, log_pi, logA):
                p.grad = None
            E = X @ Wt.t() + bias
            scores = fv.ViterbiScore.apply(log_pi, logA, E, lengths, "flash", 16)
            loss = scores.sum()
            loss.backward()
            return loss

        for _ in range(warmup):
            step()
        torch.cuda.synchronize()
        st = torch.cuda.current_stream()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        for _ in range(steps):
            loss = step()
        e1.record(st)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / steps
        state_steps = int(lengths.astype(np.int64).sum()) * w["K"]
        # the decode alone (FLASH P=16) on the same emission scores
        with torch.no_grad():
            E = X @ Wt.t() + bias
        m = fv.Model(log_pi.detach(), logA.detach(), device=device)
        bt = fv.Batch(lengths, E=E.reshape(-1), models=[m], device=device)
        d = fv.Decoder([m], bt, mode="flash", P=16)
        d(check=True)
        lib = fv._lib.load()
        dms, _ = time_decoder(d, steps, 2, lib)
        dpi, dA, _ = fv.backward(m, bt, d.paths, torch.ones(bt.n, device=device))
        for _ in range(2):
            fv.backward(m, bt, d.paths, torch.ones(bt.n, device=device))
        torch.cuda.synchronize()
        e0.record(st)
        for _ in range(steps):
            fv.backward(m, bt, d.paths, torch.ones(bt.n, device=device))
        e1.record(st)
        torch.cuda.synchronize()
        bms = e0.elapsed_time(e1) / steps
        # exactness of the count gradient: sum dlogA = sum_b (T_b - 1), sum dlog_pi = n (g = 1)
        sums_exact = bool(float(dA.double().sum()) == float((lengths.astype(np.int64) - 1).sum())
                          and float(dpi.double().sum()) == float(len(lengths)))
        return {"workload": "512 sequences, T in [20, 512], K=128 tags, 256 features; E = X W^T + b",
                "ms_per_train_step": ms, "value": state_steps / (ms / 1e3), "unit": UNIT,
                "decode_flash_P16_ms": dms, "backward_ms": bms, "loss": float(loss.item()),
                "count_gradient_sums_exact": sums_exact, "engine_variant": tuned,
                "note": "train step = emission GEMM + FLASH decode + path-count backward + GEMM gradients, "
                        "through torch.autograd (host work included)"}
    finally:
        torch.backends.cuda.matmul.allow_tf32 = prev_tf32


def er_sweep(fv, device, reps=3):
    """The paper's Erdos-Renyi family (Sec. VI): one sequence per point,
    discrete emissions over 50 symbols; decode time (CUDA events, mean of
    reps after warm-up) and decoder workspace per mode.  Sweeps: p at
    K=T=512; K at p=0.253, T=512; T at p=0.253, K=512; beam width at K=2048,
    T=512 (FLASH-BS P=16, with the relative score gap to the exact path)."""
    import torch

    import workloads as W
    st = torch.cuda.current_stream()

    def timed(d):
        d(check=True)
        for _ in range(2):
            d.launch()
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(st)
        for _ in range(reps):
            d.launch()
        e1.record(st)
        torch.cuda.synchronize()
        assert d.device_status() == 0
        return e0.elapsed_time(e1) / reps

    def point(K, T, p, modes, seed):
        c = W.erdos_renyi_case(K, T, p, seed=seed)
        m = fv.Model(c["log_pi"], c["logA"], logB=c["logB"], device=device)
        b = fv.Batch([T], obs=c["obs"], models=[m], device=device)
        out = {"K": K, "T": T, "p": round(p, 6)}
        ref = None
        for name, kw in modes:
            d = fv.Decoder([m], b, **kw)
            row = {"ms": timed(d), "workspace_bytes": d.ws_bytes}
            s = float(d.scores[0].item())
            if ref is None:
                ref = (d.paths[:T].clone(), s)
            else:
                row["same_path_as_vanilla"] = bool(torch.equal(ref[0], d.paths[:T]))
                row["score_gap"] = abs(ref[1] - s) / abs(ref[1]) if ref[1] else 0.0
            out[name] = row
            del d
        return out

    def exact_modes(K):
        return (("vanilla", {"mode": "vanilla"}), ("flash_P16", {"mode": "flash", "P": 16}),
                ("flash_bs_P16_fullwidth", {"mode": "beam", "B": K, "P": 16}))

    D = W.ER_DEFAULT
    res = {"workload": "Erdos-Renyi HMMs (edge probability p, absent edges -inf), 50 symbols, one sequence",
           "p_sweep": [point(D["K"], D["T"], p, exact_modes(D["K"]), 100 + i) for i, p in enumerate(W.ER_P_SWEEP)],
           "K_sweep": [point(K, D["T"], D["p"], exact_modes(K), 200 + i) for i, K in enumerate(W.ER_SIZE_SWEEP)],
           "T_sweep": [point(D["K"], T, D["p"], exact_modes(D["K"]), 300 + i) for i, T in enumerate(W.ER_SIZE_SWEEP)]}
    res["B_sweep"] = point(2048, D["T"], D["p"], (("vanilla", {"mode": "vanilla"}),) + tuple(
        (f"flash_bs_P16_B{B}", {"mode": "beam", "B": B, "P": 16}) for B in W.ER_BEAM_SWEEP), 400)
    return res


def config3_dense(fv, T, device, lib):
    """K=4096 dense (Dirichlet 0.1 rows), batch 8 of length T: vanilla with
    the full backpointer table against FLASH P=16 under a backpointer budget
    of 1/16 of that table (budget leaves)."""
    import torch

    import workloads as W
    K, n = 4096, 8
    log_pi, logA = W.config3_dense_model()
    m = fv.Model(log_pi, logA, device=device)
    E = W.gaussian_emissions_packed_device(n * T, K, seed=3, device=device, chunk_rows=1 << 16)
    b = fv.Batch([T] * n, E=E.view(-1), models=[m], device=device)
    table = n * T * K * 2
    out = {"workload": f"K={K} dense (Dirichlet 0.1 rows), batch {n}, T={T}, E = log_softmax N(0,1)",
           "state_steps": n * T * K}
    res = {}
    for name, kw in (("vanilla", {"mode": "vanilla"}),
                     ("flash_P16_budget_1_16", {"mode": "flash", "P": 16, "mem_budget": table // 16}),
                     ("checkpoint_sqrtT", {"mode": "checkpoint", "P": 0})):
        d = fv.Decoder([m], b, **kw)
        d(check=True)
        ms, fwd = time_decoder(d, 1, 0, lib)
        res[name] = d
        out[name] = {"ms": ms, "value": n * T * K / (ms / 1e3), "unit": UNIT, "workspace_bytes": d.ws_bytes,
                     "forward_kernels_ms": fwd}
    ph = flash_phases(res["flash_P16_budget_1_16"], lib)
    ph["leaf_waves_ms"] = ph["task_level_ms"][-1] if ph["task_level_ms"] else None
    ph["root_vs_vanilla_forward"] = ph["root_pass_ms"] / out["vanilla"]["forward_kernels_ms"]
    out["flash_P16_budget_1_16"]["phases"] = ph
    pv, sv = res["vanilla"].paths, res["vanilla"].scores
    pf, sf = res["flash_P16_budget_1_16"].paths, res["flash_P16_budget_1_16"].scores
    out["flash_P16_budget_1_16"]["bit_identical_to_vanilla"] = bool(
        torch.equal(pv, pf) and torch.equal(sv.view(torch.int32), sf.view(torch.int32)))
    out["flash_P16_budget_1_16"]["time_vs_vanilla"] = out["flash_P16_budget_1_16"]["ms"] / out["vanilla"]["ms"]
    out["flash_P16_budget_1_16"]["leaf_budget_bytes"] = table // 16
    pc_, sc_ = res["checkpoint_sqrtT"].paths, res["checkpoint_sqrtT"].scores
    out["checkpoint_sqrtT"]["bit_identical_to_vanilla"] = bool(
        torch.equal(pv, pc_) and torch.equal(sv.view(torch.int32), sc_.view(torch.int32)))
    out["checkpoint_sqrtT"]["time_vs_vanilla"] = out["checkpoint_sqrtT"]["ms"] / out["vanilla"]["ms"]
    out["full_backpointer_table_bytes"] = table
    cells = n * (T - 1) * K * K
    pk, _ = peaks()
    peak = measured_alu_peak(fv)["tflops"]
    lane_peak = alu_peak_tops(pk.get("sm_max_mhz", 2070.0), sm_count(device))
    fwd = out["vanilla"]["forward_kernels_ms"]
    achieved = 2.0 * cells / (fwd / 1e3) / 1e12
    # the bounded-row engine forms a share of the K^2 candidates and reads
    # that share of logA, so this is the rate of the full recursion it stands for
    out["full_recursion_equivalent"] = {"kernel": "prune_fwd_kernel", "bound": "latency and L2 reads of rows",
                                        "tflops": achieved, "of_measured_maxplus_peak": achieved / peak,
                                        "of_fp32_lanes": achieved / lane_peak, "kernel_ms": fwd, "cells": cells}
    del res, E
    torch.cuda.empty_cache()
    return out


def config3_sparse(fv, T, device, lib):
    """K=65536 CSR (32 successors per state), batch 8 of length T: dynamic
    beam search with B in {128, 512, 2048}.  The emission scores of all 8
    sequences (8 T K floats: 210 GB at T = 100 000) are drawn on the device
    once and every beam width decodes them; when they do not fit next to
    the decoder, the batch runs in rounds of fewer sequences (the times add
    up)."""
    import torch

    import workloads as W
    K, n = 65536, 8
    log_pi, rp, col, val = W.config3_sparse_model()
    m = fv.Model(log_pi, row_ptr=rp, col=col, val=val, device=device)
    torch.cuda.empty_cache()
    rounds = None
    for per_round in (8, 4, 2, 1):
        try:
            E = W.gaussian_emissions_packed_device(per_round * T, K, seed=4, device=device, chunk_rows=1 << 13)
            # room for the largest decoder workspace next to E
            probe = fv.workspace_size([m], fv.Batch([T] * per_round, E=E.view(-1), models=[m], device=device),
                                      mode="beam", B=2048, P=0)
            spare = torch.empty(probe, dtype=torch.uint8, device=device)
            del spare
            rounds = per_round
            break
        except torch.cuda.OutOfMemoryError:
            E = None
            torch.cuda.empty_cache()
    out = {"workload": f"K={K} CSR (32 successors, Dirichlet 1 weights), batch {n}, T={T}, E = log_softmax N(0,1)",
           "sequences_per_round": rounds,
           "note": "with fewer than 8 sequences per round every round decodes the same seeded rows and the "
                   "times are per-round time x rounds"}
    b = fv.Batch([T] * rounds, E=E.view(-1), models=[m], device=device)
    hbm = peaks()[0].get("hbm_gbs", 6800.0)
    for B in (128, 512, 2048):
        d = fv.Decoder([m], b, mode="beam", B=B, P=0)
        d(check=True)
        ms_round, fwd = time_decoder(d, 1, 0, lib)
        ms = ms_round * (n // rounds)
        eps = n * (T - 1) * B * 32 / (ms / 1e3)
        # algorithmic bytes per edge relaxation: column index + edge weight,
        # plus the emission score of its target (an upper bound: targets
        # reached twice are read once)
        gbs = 12.0 * eps / 1e9
        out[f"beam_B{B}"] = {"ms": ms, "value": n * T * K / (ms / 1e3), "unit": UNIT,
                             "ms_per_step": ms / T, "edge_relaxations_per_s": eps, "workspace_bytes": d.ws_bytes,
                             "engine": "cluster of 8 CTAs per sequence" if B >= 64 else "one CTA per sequence",
                             "roofline": {"bound": "latency", "achieved": gbs, "peak": hbm, "unit": "GB/s",
                                          "frac": gbs / hbm, "bytes_per_edge": 12,
                                          "note": "per-step latency (cluster barriers of the top-B select), "
                                                  "not bandwidth, bounds the step"}}
        del d
    del E, b
    torch.cuda.empty_cache()
    return out


def candidate_share(log_pi, logA, E, K, steps=256, warm=32):
    """Share of the K^2 candidates of a step that the bounded-row engine's
    bounds leave: the listed weights of a column and, per warp of columns, the
    rows whose delta could still pass a column's maximum.  Counted over steps
    warm .. steps of the first sequence (E: its rows), with the maxima known;
    the engine forms a few more, since it starts from a depth it expects."""
    import torch
    M = 6 if K <= 256 else 12 if K <= 512 else 16 if K <= 1024 else 32
    warp = 64 if K <= 256 else 128  # columns of a warp
    A = torch.as_tensor(logA, dtype=torch.float32, device=E.device)
    cut = A.topk(M + 1, dim=0).values[M]
    d = torch.as_tensor(log_pi, dtype=torch.float32, device=E.device) + E[0]
    rows, n = 0.0, 0
    for t in range(1, min(steps, E.shape[0])):
        best = (d[:, None] + A).amax(0)
        if t >= warm:
            need = torch.stack([x.min() for x in (best - cut).split(warp)])
            rows += float((d[None, :] >= need[:, None]).sum(1).float().mean())
            n += 1
        d = best + E[t]
    return min(1.0, (M + rows / max(n, 1)) / K)


def larger_k_rows(fv, device, lib, peak_tflops, Ks=(512, 1024), n_seq=256):
    """Exact decoding at larger state spaces: 256 sequences, T uniform in
    [500, 4000], Dirichlet(1) rows, log-softmax emissions; forward-kernel
    time, the candidates it forms against the measured max-plus ceiling, and
    the rate of the full recursion it stands for."""
    import torch

    import workloads as W
    rows = {}
    for K in Ks:
        log_pi, logA = W.config2_model(seed=2, K=K)
        lengths = W.config2_lengths(seed=2, n_seq=n_seq)
        E = W.gaussian_emissions_packed_device(int(lengths.sum()), K, seed=2, device=device)
        m = fv.Model(log_pi, logA, device=device)
        b = fv.Batch(lengths, E=E.view(-1), models=[m], device=device)
        d = fv.Decoder([m], b, mode="vanilla")
        d(check=True)
        ms, fwd = time_decoder(d, 3, 2, lib)
        cells = int((lengths.astype(np.int64) - 1).sum()) * K * K
        achieved = 2.0 * cells / (fwd / 1e3) / 1e12
        share = candidate_share(log_pi, logA, E.view(-1, K)[:int(lengths[0])], K)
        rows[f"K{K}"] = {"workload": f"{n_seq} sequences, K={K} dense FP32, T~U[500,4000]",
                         "ms": ms, "value": int(lengths.sum()) * K / (ms / 1e3), "unit": UNIT,
                         "roofline": {"bound": "latency and L2 reads of rows",
                                      "achieved": achieved * share, "peak": peak_tflops, "unit": "TFLOP/s",
                                      "frac": achieved * share / peak_tflops, "kernel_ms": fwd, "candidate_share": share,
                                      "full_recursion_equivalent_tflops": achieved}}
        del d, b, E
        torch.cuda.empty_cache()
    return rows


def static_vs_dynamic_beam(fv, device, lib):
    """The static beam the paper contrasts with its dynamic one (Sec. II-B,
    Sec. V-C.1) against the dynamic beam, same inputs, same results: time per
    decode and the candidate storage each step needs (static: the score and
    source of all K states, in the workspace; dynamic: only the states the
    beam reaches, listed in shared memory for CSR)."""
    import torch

    import workloads as W
    rows = {}
    cases = []
    rng = np.random.default_rng(77)
    log_pi, logA = W.random_model(1024, rng)
    md = fv.Model(log_pi, logA, device=device)
    Ed = torch.from_numpy(W.gaussian_emissions(64 * 2000, 1024, rng)).to(device)
    cases.append(("dense_K1024_B256_64x2000", md, fv.Batch([2000] * 64, E=Ed.view(-1), models=[md], device=device),
                  256, 1024))
    log_pi, rp, col, val = W.config3_sparse_model()
    ms = fv.Model(log_pi, row_ptr=rp, col=col, val=val, device=device)
    Es = W.gaussian_emissions_packed_device(8 * 500, 65536, seed=4, device=device, chunk_rows=1 << 13)
    bs = fv.Batch([500] * 8, E=Es.view(-1), models=[ms], device=device)
    for B in (128, 512, 2048):
        cases.append((f"csr_K65536_B{B}_8x500", ms, bs, B, 65536))
    for name, m, b, B, K in cases:
        row = {}
        res = {}
        for kind, flags in (("dynamic", 0), ("static", fv._lib.FV_STATIC_BEAM)):
            d = fv.Decoder([m], b, mode="beam", B=B, P=0, flags=flags)
            d(check=True)
            ms_, _ = time_decoder(d, 3, 1, lib)
            res[kind] = (d.paths.clone(), d.scores.clone())
            row[kind] = {"ms": ms_, "workspace_bytes": d.ws_bytes}
            del d
        row["static"]["candidate_bytes_per_step"] = 8 * K
        row["dynamic"]["candidate_bytes_per_step"] = 8 * (min(K, 32 * B) if K == 65536 else K)
        row["static_over_dynamic_time"] = row["static"]["ms"] / row["dynamic"]["ms"]
        row["identical"] = bool(torch.equal(res["static"][0], res["dynamic"][0]) and torch.equal(
            res["static"][1].view(torch.int32), res["dynamic"][1].view(torch.int32)))
        rows[name] = row
    del Ed, Es
    torch.cuda.empty_cache()
    return rows


def serving_run(seconds, rate=2000.0, n_streams=64, max_wall=None):
    """Serving loop: Poisson arrivals, mixed K and T, exact and beam B=256,
    admitted under a 40 GB device-memory budget and packed per class (K,
    mode) into shared launches; one served model per K class, emission
    scores drawn on the device per request.  Admission stops after max_wall
    seconds (default: three times the arrival window); requests still
    waiting then are counted as not served."""
    from paper_2510_19301_gb300.serve import GpuBackend, Server, poisson_requests
    reqs = poisson_requests(rate=rate, seconds=seconds, seed=6)
    be = GpuBackend(n_streams=n_streams)
    variants = be.tune((64, 256, 1024))
    srv = Server(be, mem_budget_bytes=40 << 30, max_inflight=n_streams)
    rep = srv.run(reqs, max_wall=3 * seconds if max_wall is None else max_wall)
    rep["engine_variants"] = variants
    rep.update({"arrival_rate_req_s": rate, "arrival_window_s": seconds, "offered": len(reqs),
                "mix": "K uniform {64,256,1024}, T log-uniform [100,20000], 50% exact (vanilla) / "
                       "50% beam B=256; one served Dirichlet(1) model per K class",
                "streams": n_streams})
    return rep


def run_reference(args):
    rank, world, _ = dist_env()
    if rank != 0:
        return
    import oracle
    import workloads as W
    oracle.build()
    K = 256
    log_pi, logA = W.config2_model(seed=2)
    lengths = W.config2_lengths(seed=2, n_seq=args.n_seq)
    hmm = oracle.HMM(log_pi, logA)
    cores = os.cpu_count() or 1
    n = cores  # one sequence per core per step: a bounded sample of the batch
    rng = np.random.default_rng(123)
    times, total = [], 0
    for it in range(args.warmup + args.steps):
        idx = [(it * n + k) % len(lengths) for k in range(n)]
        jobs = [W.gaussian_emissions(int(lengths[i]), K, rng) for i in idx]
        t0 = time.perf_counter()
        oracle.map_sequences(lambda e: oracle.viterbi(hmm, e), jobs, threads=cores)
        dt = time.perf_counter() - t0
        if it >= args.warmup:
            times.append(dt)
            total += int(sum(int(lengths[i]) for i in idx)) * K
    T = sum(times)
    v = total / T
    out = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": world,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000 * T / args.steps,
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
           "data": "synthetic",
           "config": {"workload": WORKLOAD, "mode": "vanilla", "sample_per_step": f"{n} sequences"},
           "cpu_baseline": {"value": v, "unit": UNIT, "cores": cores, "kind": "oracle",
                            "sample": f"{n} sequences of the workload per step (one per core), exact vanilla oracle"},
           "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


def run_ours(args):
    import torch
    import torch.distributed as dist

    import paper_2510_19301_gb300 as fv
    rank, world, local = dist_env()
    if world > 1:
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    torch.cuda.set_device(local)
    device = f"cuda:{local}"
    wl = make_workload(args, rank, device)
    K = wl["K"]
    lengths = wl["lengths"]
    m = wl["model"]
    batch = fv.Batch(lengths, E=wl["E"].view(-1), models=[m], device=device)
    # engine configuration for this K class picked by the autotuner on this
    # very batch (all candidates give identical results)
    if args.engine_variant >= 0:
        fv.set_engine_variant(K, args.engine_variant)
        chosen = [args.engine_variant]
    else:
        chosen = fv.autotune([m], batch, mode=args.mode, P=args.P, B=args.B, mem_budget=args.budget)
    dec = fv.Decoder([m], batch, mode=args.mode, P=args.P, B=args.B, mem_budget=args.budget)
    lib = fv._lib.load()
    state_steps = int(lengths.astype(np.int64).sum()) * K
    cells = int((lengths.astype(np.int64) - 1).sum()) * K * K

    # measured max-plus ceiling (before the timed region)
    alu_probe = measured_alu_peak(fv)

    # correctness gate of the timed configuration: device status must be OK
    dec(check=True)
    for _ in range(args.warmup):
        dec.launch()
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    clk = ClockSampler(local)
    clk.start()
    lib.fv_timing_enable(1)
    st = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(st)
    for _ in range(args.steps):
        dec.launch()
    e1.record(st)
    torch.cuda.synchronize()
    if world > 1:
        dist.barrier()
    clocks = clk.stop()
    ms = e0.elapsed_time(e1) / args.steps
    import ctypes
    tot = ctypes.c_float(0)
    npairs = ctypes.c_int32(0)
    lib.fv_timing_read(ctypes.byref(tot), ctypes.byref(npairs))
    lib.fv_timing_enable(0)
    fwd_ms = tot.value / max(npairs.value, 1)
    status = dec.device_status()
    assert status == 0, f"device status {status}"

    value, ms_max, _ = aggregate_ranks(ms, state_steps, device=device)

    # end to end through the public API: every step copies its emission
    # scores from pinned host memory to the device, decodes them and reads
    # paths + scores back to pinned host memory.  Two device input buffers
    # (two Decoders) let the copy for step i+1 run on a copy stream while
    # step i decodes.
    E_host = torch.empty(wl["E"].numel(), dtype=torch.float32, pin_memory=True)
    E_host.copy_(wl["E"].view(-1))
    E_dev = [batch.E, torch.empty_like(batch.E)]
    batch2 = fv.Batch(lengths, E=E_dev[1], models=[m], device=device)
    decs = [dec, fv.Decoder([m], batch2, mode=args.mode, P=args.P, B=args.B, mem_budget=args.budget)]
    P_host = [torch.empty(dec.paths.numel(), dtype=torch.int32, pin_memory=True) for _ in range(2)]
    S_host = [torch.empty(dec.scores.numel(), dtype=torch.float32, pin_memory=True) for _ in range(2)]
    copy_st = torch.cuda.Stream(device=device)
    d2h_st = torch.cuda.Stream(device=device)
    # the input copy alone (the pipelined step cannot be shorter than this
    # or than the decode), best of three
    h2d_alone_ms = float("inf")
    for _ in range(3):
        torch.cuda.synchronize()
        h0, h1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        h0.record(copy_st)
        with torch.cuda.stream(copy_st):
            E_dev[1].copy_(E_host, non_blocking=True)
        h1.record(copy_st)
        torch.cuda.synchronize()
        h2d_alone_ms = min(h2d_alone_ms, h0.elapsed_time(h1))
    copied = [torch.cuda.Event() for _ in range(2)]
    consumed = [torch.cuda.Event() for _ in range(2)]
    returned = [torch.cuda.Event() for _ in range(2)]
    e2e_steps = max(3, min(args.steps, 20))
    f0 = torch.cuda.Event(enable_timing=True)
    f1 = torch.cuda.Event(enable_timing=True)
    for it in range(1 + e2e_steps):
        if it == 1:
            torch.cuda.synchronize()
            f0.record(st)
            copy_st.wait_event(f0)
        k = it % 2
        copy_st.wait_event(consumed[k])  # the decode that last read this buffer is done
        with torch.cuda.stream(copy_st):
            E_dev[k].copy_(E_host, non_blocking=True)
        copied[k].record(copy_st)
        st.wait_event(copied[k])
        st.wait_event(returned[k])  # this decoder's previous results are read back
        decs[k].launch(st)
        consumed[k].record(st)
        # results go back on their own stream, so the next decode does not
        # queue behind them (or behind the next input copy)
        d2h_st.wait_event(consumed[k])
        with torch.cuda.stream(d2h_st):
            P_host[k].copy_(decs[k].paths, non_blocking=True)
            S_host[k].copy_(decs[k].scores, non_blocking=True)
        returned[k].record(d2h_st)
    st.wait_stream(d2h_st)
    f1.record(st)
    torch.cuda.synchronize()
    e2e_ms = f0.elapsed_time(f1) / e2e_steps
    e2e_value, _, _ = aggregate_ranks(e2e_ms, state_steps, device=device)
    h2d = E_host.numel() * 4
    d2h = P_host[0].numel() * 4 + S_host[0].numel() * 4
    assert decs[0].device_status() == 0 and decs[1].device_status() == 0
    assert torch.equal(decs[0].paths, decs[1].paths)
    del decs[1], batch2, E_dev[1]

    modes = {}
    if not args.quick:
        for P in (4, 16, 64):
            dflash = fv.Decoder([m], batch, mode="flash", P=P)
            dflash(check=True)
            fms, fk = time_decoder(dflash, max(2, args.steps // 20), 2, lib)
            modes[f"flash_P{P}"] = {"value": state_steps / (fms / 1e3), "unit": UNIT, "ms_per_step": fms,
                                   "time_vs_vanilla": fms / ms, "bit_identical_to_vanilla": None}
            pv_, sv_ = dec.paths.clone(), dec.scores.clone()
            pf_, sf_ = dflash.paths, dflash.scores
            modes[f"flash_P{P}"]["bit_identical_to_vanilla"] = bool(
                torch.equal(pv_, pf_) and torch.equal(sv_.view(torch.int32), sf_.view(torch.int32)))
            del dflash
        # budget leaves: FLASH P=16 whose leaf backpointers fit 1/16 of the
        # full table
        table = int(lengths.astype(np.int64).sum()) * K * 2
        db = fv.Decoder([m], batch, mode="flash", P=16, mem_budget=table // 16)
        db(check=True)
        bms, _ = time_decoder(db, max(2, args.steps // 20), 2, lib)
        ph = flash_phases(db, lib)
        ph["leaf_waves_ms"] = ph["task_level_ms"][-1] if ph["task_level_ms"] else None
        ph["root_vs_vanilla"] = ph["root_pass_ms"] / fwd_ms if ph["root_pass_ms"] else None
        modes["flash_P16_budget_1_16"] = {
            "phases": ph,
            "value": state_steps / (bms / 1e3), "unit": UNIT, "ms_per_step": bms, "time_vs_vanilla": bms / ms,
            "bit_identical_to_vanilla": bool(torch.equal(dec.paths, db.paths) and torch.equal(
                dec.scores.view(torch.int32), db.scores.view(torch.int32))),
            "workspace_bytes": db.ws_bytes, "vanilla_workspace_bytes": dec.ws_bytes,
            "full_backpointer_table_bytes": table, "leaf_budget_bytes": table // 16}
        del db
        # Checkpoint Viterbi (the sqrt(T)-checkpoint baseline of Sec. II-A)
        dc = fv.Decoder([m], batch, mode="checkpoint", P=0)
        dc(check=True)
        cms, _ = time_decoder(dc, max(2, args.steps // 20), 2, lib)
        modes["checkpoint_sqrtT"] = {
            "value": state_steps / (cms / 1e3), "unit": UNIT, "ms_per_step": cms, "time_vs_vanilla": cms / ms,
            "bit_identical_to_vanilla": bool(torch.equal(dec.paths, dc.paths) and torch.equal(
                dec.scores.view(torch.int32), dc.scores.view(torch.int32))),
            "workspace_bytes": dc.ws_bytes, "vanilla_workspace_bytes": dec.ws_bytes,
            "note": "ceil(sqrt T) delta checkpoints per sequence, then one engine launch per checkpoint level "
                    "re-decoding the latest segment of every sequence"}
        del dc
        comp = per_sequence_comparator(fv, m, lengths, wl["E"], K, 32, device)
        comp["batched_over_per_sequence"] = value / world / comp["value"]
        modes["plain_per_sequence_gpu"] = comp

    pk, pk_kind = peaks()
    sms = sm_count(device)
    lane_peak = alu_peak_tops(pk.get("sm_max_mhz", 2070.0), sms)
    peak = alu_probe["tflops"]
    achieved = 2.0 * cells / (fwd_ms / 1e3) / 1e12
    # vanilla: prep, order, (model preparation,) forward, trace and its repair
    bounded = args.mode == "vanilla" and int(chosen[0]) == 0
    # (above K = 256 also the launches for sequences handed to the other engines)
    launches = args.steps * ((9 if K > 256 else 6 if K > 128 else 5) if bounded else 4)
    share = 1.0
    if bounded and K > 128:
        share = candidate_share(wl["log_pi"], wl["logA"], wl["E"].view(-1, K)[:int(lengths[0])], K)

    wl_name = WORKLOAD if (args.K == 256 and args.n_seq == 1024) else WORKLOAD.replace(
        "1024 seqs, K=256", f"{args.n_seq} seqs, K={args.K}")
    out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
           "warmup": args.warmup, "ms_per_step": ms_max, "higher_is_better": True, "scaling": "weak",
           "vs_baseline": None, "dtype": "f32", "data": "synthetic",
           "config": {"workload": wl_name, "mode": args.mode, "P": args.P, "B": args.B,
                      "n_seq": int(len(lengths)), "sum_T": int(lengths.sum()), "K": K,
                      "engine_variant": int(chosen[0]),
                      "l2": "inputs larger than L2 (E is %.2f GB per step)" % (wl["E"].numel() * 4 / 1e9)},
           "clocks": clocks,
           "gpu_launches": launches,
           "roofline": {"bound": "latency" if bounded else "alu",
                        "kernel": "prune_fwd_kernel" if bounded and K > 128 else
                                  "small_value_kernel" if bounded else "dense_fwd_kernel",
                        "achieved": achieved * share,
                        "peak": peak, "unit": "TFLOP/s", "frac": achieved * share / peak,
                        "candidate_share": share,
                        "candidate_note": "share of the K^2 candidates per step that the engine's bounds leave, counted "
                                          "on the first sequence (the others cannot win); achieved counts those, "
                                          "full_recursion_equivalent_tflops all",
                        "full_recursion_equivalent_tflops": achieved,
                        "traffic": (DRAM_BYTES_PER_STATE_STEP * state_steps
                                    if (args.K == 256 and args.mode == "vanilla" and int(chosen[0]) == TRAFFIC_VARIANT)
                                    else None),
                        "traffic_note": "dram__bytes_read.sum + dram__bytes_write.sum of one ncu capture of "
                                        "this kernel (default configuration) on 608 sequences (%.2f B per "
                                        "state-step), scaled to this launch's state-steps; null for another "
                                        "configuration" % DRAM_BYTES_PER_STATE_STEP,
                        "peak_kind": "measured: fv_maxplus_peak, the engines' add + 3-input max cell on every SM "
                                     "(%.1f cells/clk/SM, 2 ops per cell)" % alu_probe["cells_per_clk_per_sm"],
                        "sm_count": sms,
                        "peak_fp32_lanes": lane_peak,
                        "frac_of_fp32_lanes": achieved * share / lane_peak,
                        "peak_fp32_lanes_kind": "derived: %d SMs x 128 FP32 lanes x 2 ops x %.0f MHz (max clock); "
                                                "the FP32 max runs at half the add rate, so no max-plus code "
                                                "reaches it" % (sms, pk.get("sm_max_mhz", 2070.0)),
                        "ops_per_cell": 2, "cells_per_launch": cells, "kernel_ms": fwd_ms},
           "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": h2d,
                   "pipelining": "two device input buffers: the H2D copy of step i+1 overlaps the decode of step i; "
                                 "results return on a third stream",
                   "d2h_bytes_per_step": d2h, "ms_per_step": e2e_ms, "h2d_alone_ms": h2d_alone_ms,
                   "h2d_alone_gb_s": h2d / (h2d_alone_ms / 1e3) / 1e9, "decode_ms": ms}}
    if modes:
        out["modes"] = modes
    if rank == 0 and not args.quick:
        out["config1"] = config1_latency(fv, device)
        out["config4_train"] = config4_train(fv, device)
    if rank == 0 and args.c3_T > 0:
        out["config3_dense"] = config3_dense(fv, args.c3_T, device, lib)
    if rank == 0 and args.c3s_T > 0:
        out["config3_sparse"] = config3_sparse(fv, args.c3s_T, device, lib)
    if rank == 0 and not args.quick:
        out["exact_larger_k"] = larger_k_rows(fv, device, lib, alu_probe["tflops"])
        out["beam_static_vs_dynamic"] = static_vs_dynamic_beam(fv, device, lib)
    if rank == 0 and args.serve_seconds > 0:
        out["serving"] = serving_run(args.serve_seconds)
        # the same request mix at a tenth of the rate: fewer requests share a
        # launch, so the latencies are closer to one request's service time
        out["serving_low_rate"] = serving_run(5.0, rate=200.0)
    if rank == 0 and world == 1 and not args.no_cpu:
        out["cpu_baseline"] = cpu_baseline(wl)
    if rank == 0:
        print(json.dumps(out), flush=True)
    if world > 1:
        dist.destroy_process_group()


def run_er_sweep():
    import torch

    import paper_2510_19301_gb300 as fv
    torch.cuda.set_device(0)
    res = er_sweep(fv, "cuda:0")
    print(json.dumps({"metric": "Erdos-Renyi sweep: decode ms and workspace bytes per mode", "data": "synthetic",
                      "n_gpus": 1, **res}), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--mode", default="vanilla", choices=["vanilla", "flash", "beam"])
    ap.add_argument("--P", type=int, default=16)
    ap.add_argument("--B", type=int, default=0)
    ap.add_argument("--budget", type=int, default=0)
    ap.add_argument("--n-seq", dest="n_seq", type=int, default=1024)
    ap.add_argument("--K", type=int, default=256, help="states (the default workload has K=256)")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--quick", action="store_true", help="skip the FLASH and per-sequence rows")
    ap.add_argument("--c3-T", dest="c3_T", type=int, default=100000,
                    help="length of the K=4096 batch-8 run (0 = skip)")
    ap.add_argument("--c3s-T", dest="c3s_T", type=int, default=100000,
                    help="length of the K=65536 sparse beam runs (0 = skip)")
    ap.add_argument("--engine-variant", dest="engine_variant", type=int, default=-1,
                    help="engine configuration of the K class (default: picked by the autotuner)")
    ap.add_argument("--er-sweep", dest="er_sweep", action="store_true",
                    help="only the Erdos-Renyi sweep of the paper's synthetic family (one JSON line)")
    ap.add_argument("--serve-seconds", dest="serve_seconds", type=float, default=60.0,
                    help="arrival window of the serving run (default: the full 60 s serving workload; 0 = skip)")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.impl == "reference":
        run_reference(args)
    elif args.er_sweep:
        run_er_sweep()
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
