#!/usr/bin/env python
"""Benchmark of the fused NBM training step (arXiv 2210.14907, Sec. 3).

One step = sample 262,144 collocation points -> cut-cell geometry -> two-network
7-point stencil forward (BF16 tcgen05 hidden GEMMs) -> FV balance / jump rows
-> squared loss -> backward -> Adam, on the sphere-interface workload with
h = 2/128 and two 3->128->128->128->1 tanh networks (the mixed-precision
configuration).  Prints one JSON line (rank 0).

  python bench.py [--steps K] [--warmup W] [--gpus N] [--impl ours|reference]

Timing: every timed step is bracketed by CUDA events on the launching stream;
L2 is flushed (256 MiB write) between timed steps, outside the events.  The
fused kernel is additionally timed live (libnbm's event profiler) for the
roofline line.  Under torchrun (N > 1) the step is data parallel (Sec. 3:
points distributed over the GPUs, gradients aggregated): every rank takes its
262,144-point shard of an N x 262,144-point batch (weak scaling), the gradient
and the loss are summed over the ranks by NCCL all-reduce, and every rank
applies the same Adam update; the reported time is the max over ranks.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = ("collocation pts/sec per train step (mixed vs FP32, same L∞ err); "
          "% tensor peak")
UNIT = "collocation points/s"
WORKLOAD = ("sphere interface (r0=0.5, mu-=1, mu+=10), h=2/128, 262144 uniform collocation "
            "points per step, two 3->128->128->128->1 tanh MLPs, BF16 tcgen05 hidden GEMMs "
            "with FP32 accumulate, Adam lr 1e-3")
BATCH = 262_144
# DRAM bytes (read + write) per launch of the fused kernel, from an ncu capture
# of that kernel on this workload, with the SHA-256 (first 16 hex digits) of
# the kernel's sources at the time of the capture.  The bench line reports the
# figure only while the sources still hash to that value (else null).
FUSED_TRAFFIC = {"bytes": 9_057_280, "sources_sha16": "ed8f503dc26c47fb"}
FUSED_SOURCES = ("paper_2210_14907_gb300/csrc/nbm_tc.cu", "paper_2210_14907_gb300/csrc/nbm_tc_layer.cuh",
                 "paper_2210_14907_gb300/csrc/nbm_tc_ptx.cuh", "paper_2210_14907_gb300/csrc/nbm_device.cuh")
# libnbm kernel launches per timed step.  One nbm_train_steps call of one C2
# step: k_sample_classify (its extra blocks restage the weights), k_scatter
# (up to 2048 blocks of points it also does the block-count scan, so no
# k_scan_counts; it writes the uncut points' tile records); k_cut_geometry
# (the cut cells' records); k_fwd_tc (cut-cell forward), k_cut_residual;
# k_step_tc (fused train step); k_reduce_adam (loss, gradient, update).  The
# data-parallel step (N > 1) runs the same chain through nbm_loss_grad_shard
# (k_reduce_adam writes the loss and gradient only) and then k_adam: one more.
# (Batches above 2048 blocks of 256 points, such as the 1M-point secondary
# workload, add k_scan_counts and k_gather_tiles, which writes the records.)
LAUNCHES_PER_STEP = 7
LAUNCHES_PER_DP_STEP = 8
# FP32 FFMA peak of the plain path's roofline: 152 SMs x 128 FP32 lanes x
# 2 FLOP per FMA x the SM clock (GB300's 2070 MHz maximum, the clock the
# timed region ran at).
SMS, FP32_LANES, SM_MAX_MHZ = 152, 128, 2070.0


def fused_sources_sha16():
    h = hashlib.sha256()
    for f in FUSED_SOURCES:
        with open(os.path.join(ROOT, f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            d = json.load(f)
        return d["bf16_tflops"], d["bf16_tflops_sustained"], d["hbm_gbs"], "measured"
    except Exception:
        return 1900.0, 1700.0, 6800.0, "fallback"


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.idx = str(gpu_index)
        self.rows = []
        self.proc = None
        self.mark = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                 "-lms", "100"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
            return
        self.t = threading.Thread(target=self._read, daemon=True)
        self.t.start()

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 9 and parts[0] == self.idx:
                self.rows.append((time.time(), parts))

    def begin(self):
        self.mark = time.time()

    def end(self):
        self.mark_end = time.time()

    def stop(self):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()

    def summary(self):
        rows = [p for (t, p) in self.rows if self.mark and self.mark <= t <= self.mark_end + 0.05]
        if not rows:
            rows = [p for (_, p) in self.rows[-5:]]
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}

        def num(s):
            try:
                return float(s)
            except ValueError:
                return None
        sm = [num(r[1]) for r in rows if num(r[1]) is not None]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in rows for i in range(4) if r[5 + i] == "Active"})
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": num(rows[0][2]), "samples": len(rows),
                "power_w_max": max((num(r[3]) or 0.0) for r in rows), "reasons": reasons}


def _dist(gpu=True):
    """World size, rank and local rank from torchrun's environment.  Several
    ranks join one process group: gloo for host tensors (barrier, timing) and,
    when gpu is set, NCCL for device tensors (the gradient exchange), with
    NVLink SHARP (multicast) off."""
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if ws > 1:
        import torch.distributed as dist
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        os.environ.setdefault("NCCL_NVLS_ENABLE", "0")
        dist.init_process_group("cpu:gloo,cuda:nccl" if gpu else "gloo", rank=rank,
                                world_size=ws)
    return ws, rank, local


def _barrier(ws):
    """All ranks meet here (a host all-reduce over gloo)."""
    if ws > 1:
        import torch
        import torch.distributed as dist
        dist.all_reduce(torch.zeros(1))


def _max_over_ranks(ws, x):
    if ws == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def cpu_baseline(target_s=10.0, steps=1, warmup=0):
    """The FP64 oracle (OpenMP over points, all host cores) on a bounded sample
    of the C2 workload.  One step = the oracle's loss + gradient + Adam on a
    sub-batch of sampled points (counter = the step's index).  The sub-batch is
    sized so that `steps` timed steps take about target_s seconds; `warmup`
    untimed steps come first."""
    import numpy as np

    from oracle import pyoracle as O
    O.build()
    pr = O.make_problem(geometry=O.GEOM_SPHERE, n_hidden=3, width=128, mu_minus=1.0,
                        mu_plus=10.0, h=2.0 / 128)
    P = 2 * O.params_per_net(pr)
    rng = np.random.default_rng(0)
    th = rng.uniform(-0.1, 0.1, P)
    m = np.zeros(P)
    v = np.zeros(P)

    def step(t, n):
        pts = O.sample_points(pr, 1, t, n, 0)
        _, g = O.loss_grad(pr, th, pts)
        O.adam_step(th, m, v, g, t)

    t0 = time.perf_counter()
    step(1, 1024)
    t1 = time.perf_counter() - t0
    n = int(min(BATCH, max(256, 1024 * target_s / (steps * max(t1, 1e-4)))))
    for k in range(warmup):
        step(2 + k, n)
    t0 = time.perf_counter()
    for k in range(steps):
        step(2 + warmup + k, n)
    t = time.perf_counter() - t0
    cores = O.default_threads()
    return {"value": steps * n / t, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"{n} sampled points of the {BATCH}-point step (loss, gradient, Adam) "
                      f"x {steps} steps after {warmup} warm-up, FP64 oracle, OpenMP {cores} "
                      f"threads, {t:.1f} s",
            "sub_batch": n, "ms_per_step": 1e3 * t / steps, "timed_s": t}


def sphere_exact(x):
    """Manufactured solution of the sphere workload (u- inside r <= 1/2, u+ outside)."""
    import numpy as np
    r = np.sqrt((x ** 2).sum(1))
    um = np.exp(x[:, 0]) * np.cos(x[:, 1]) * np.sin(x[:, 2])
    return np.where(r <= 0.5, um, (x ** 2).sum(1))


def sec41_exact(x):
    """Manufactured solution of the Sec. 4.1 study (u- = e^z inside r <= 1/2,
    u+ = cos x sin y outside)."""
    import numpy as np
    r = np.sqrt((x ** 2).sum(1))
    return np.where(r <= 0.5, np.exp(x[:, 2]), np.cos(x[:, 0]) * np.sin(x[:, 1]))


def node_errors(u, n, exact=sphere_exact):
    """L-infinity and RMS error over the interior nodes of the (n+1)^3 grid."""
    import numpy as np
    g = -1.0 + np.arange(n + 1) * 2.0 / n
    Z, Y, X = np.meshgrid(g, g, g, indexing="ij")
    x = np.stack([X.ravel(), Y.ravel(), Z.ravel()], 1)
    e = np.abs(np.asarray(u, np.float64) - exact(x)).reshape(n + 1, n + 1, n + 1)
    e = e[1:-1, 1:-1, 1:-1]
    return float(e.max()), float(np.sqrt((e ** 2).mean()))


def trilinear(u, n, x):
    import numpy as np
    U = np.asarray(u, np.float64).reshape(n + 1, n + 1, n + 1)
    t = (x + 1.0) * n / 2.0
    i0 = np.clip(np.floor(t).astype(int), 0, n - 1)
    f = t - i0
    out = np.zeros(len(x))
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                w = ((f[:, 0] if dx else 1 - f[:, 0]) * (f[:, 1] if dy else 1 - f[:, 1])
                     * (f[:, 2] if dz else 1 - f[:, 2]))
                out += w * U[i0[:, 2] + dz, i0[:, 1] + dy, i0[:, 0] + dx]
    return out


def accuracy(dev, steps=2000):
    """The metric's accuracy half: the mixed (BF16) and the plain FP32 training step,
    each run for the workload's 2000 Adam steps from the same start, then the
    exact-solution error at the 129^3 nodes; and what the trained surrogate gains
    over the plain method (the grid CG solve at the same h, interpolated
    trilinearly) at random points within 2h of the interface."""
    import numpy as np
    import torch

    import paper_2210_14907_gb300 as nbm
    out = {"steps": steps, "batch": BATCH, "lr": 1e-3}
    keep = None
    for prec, name in ((nbm.PREC_BF16, "mixed_bf16"), (nbm.PREC_FP32, "fp32")):
        d = nbm.config("C2", precision=prec)
        prob = nbm.Problem(d)
        params = nbm.xavier_init(d, seed=0, device=dev)
        m = torch.zeros_like(params)
        v = torch.zeros_like(params)
        hist = torch.zeros(steps, device=dev)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        prob.train_steps(params, m, v, 0, steps, BATCH, lr=1e-3, seed=1, loss_hist=hist)
        torch.cuda.synchronize()
        wall = time.perf_counter() - t0
        u = prob.eval_grid(params, 128, precision=nbm.PREC_FP32).cpu().numpy()
        linf, rmse = node_errors(u, 128)
        out[name] = {"linf": linf, "rmse": rmse, "final_loss": float(hist[-50:].mean()),
                     "train_s": wall}
        if prec == nbm.PREC_BF16:
            keep = (prob, params)
    out["mixed_over_fp32_linf"] = out["mixed_bf16"]["linf"] / out["fp32"]["linf"]
    # implicit refinement (the paper's base 64^3 cells refined onto 128^3, 256^3,
    # 512^3): the same network, points and steps, every point with four cells
    d = nbm.config("C2")
    d.h, d.refine_levels = 2.0 / 64, 3
    prob = nbm.Problem(d)
    params = nbm.xavier_init(d, seed=0, device=dev)
    m = torch.zeros_like(params)
    v = torch.zeros_like(params)
    hist = torch.zeros(steps, device=dev)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    prob.train_steps(params, m, v, 0, steps, BATCH, lr=1e-3, seed=1, loss_hist=hist)
    torch.cuda.synchronize()
    wall = time.perf_counter() - t0
    u = prob.eval_grid(params, 128, precision=nbm.PREC_FP32).cpu().numpy()
    linf, rmse = node_errors(u, 128)
    out["refined_mixed_bf16"] = {
        "cells": "h = 2/64 refined onto 2/128, 2/256, 2/512 (4 cells per point)",
        "linf": linf, "rmse": rmse, "final_loss": float(hist[-50:].mean()), "train_s": wall,
        "points_per_s": steps * BATCH / wall}
    prob, params = keep
    n = 128
    ucg, it, rr, ok = prob.grid_cg_solve(n, rtol=1e-10)
    ucg = ucg.cpu().numpy()
    rng = np.random.default_rng(0)
    dirs = rng.normal(size=(200000, 3))
    dirs /= np.linalg.norm(dirs, axis=1)[:, None]
    pts = dirs * (0.5 + rng.uniform(-4.0 / n, 4.0 / n, 200000))[:, None]
    ex = sphere_exact(pts)
    us = prob.eval_points(params, torch.from_numpy(pts.astype(np.float32)).to(dev)).cpu().numpy()
    es, eg = np.abs(us - ex), np.abs(trilinear(ucg, n, pts) - ex)
    out["gain_near_interface"] = {
        "points": "200000 random points within 2h of Gamma, h = 2/128",
        "surrogate_linf": float(es.max()), "surrogate_rmse": float(np.sqrt((es ** 2).mean())),
        "grid_cg_trilinear_linf": float(eg.max()),
        "grid_cg_trilinear_rmse": float(np.sqrt((eg ** 2).mean())),
        "surrogate_bytes": params.numel() * 4, "grid_solution_bytes": (n + 1) ** 3 * 8}
    return out


# Table 1 of the paper (Sec. 4.1, JAX on one A6000, 10,000 epochs): N -> (RMSE,
# L-infinity, seconds per epoch)
PAPER_TABLE1 = {8: (3.7e-2, 3.25e-1, 0.0306), 16: (7.1e-3, 1.10e-1, 0.056),
                32: (5.9e-3, 8.36e-2, 0.053), 64: (4.1e-3, 6.44e-2, 0.287),
                128: (2.64e-3, 3.53e-2, 2.125)}


def table1(dev, epochs, resolutions, lr=1e-3):
    """The convergence study of Sec. 4.1 (Table 1): sphere of radius 1/2,
    u- = e^z, u+ = cos x sin y, mu- = y^2 ln(x+2) + 4, mu+ = e^-z, two sine
    networks of 5 hidden layers x 10 units (982 parameters), Glorot init, Adam.
    Per resolution N (h = 2/N): one epoch is N^3 freshly drawn uniform
    collocation points in mini-batches of at most 32 x 32 x 16 (the batch size
    the paper states for its scaling runs); errors at the interior nodes of the
    (N+1)^3 grid against the exact solution of each node's side."""
    import numpy as np
    import torch

    import paper_2210_14907_gb300 as nbm
    rows = []
    for N in resolutions:
        d = nbm.ProblemDesc(geometry=nbm.GEOM_SPHERE, n_hidden=5, width=10,
                            precision=nbm.PREC_FP32, h=2.0 / N, solution=nbm.SOL_SEC41,
                            activation=nbm.ACT_SIN)
        prob = nbm.Problem(d)
        params = nbm.xavier_init(d, seed=0, device=dev)
        m = torch.zeros_like(params)
        v = torch.zeros_like(params)
        batch = min(N ** 3, 32 * 32 * 16)
        steps = epochs * ((N ** 3 + batch - 1) // batch)
        hist = torch.zeros(min(steps, 1000), device=dev)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        done, chunk = 0, 1000
        while done < steps:
            k = min(chunk, steps - done)
            prob.train_steps(params, m, v, done, k, batch, lr=lr, seed=1, loss_hist=hist[:k])
            done += k
        torch.cuda.synchronize()
        wall = time.perf_counter() - t0
        u = prob.eval_grid(params, N, precision=nbm.PREC_FP32).cpu().numpy()
        linf, rmse = node_errors(u, N, sec41_exact)
        # the plain grid method on the same rows and grid, for comparison
        ucg, it_cg, _, ok_cg = prob.grid_cg_solve(N, rtol=1e-10, max_iter=100000)
        g_linf, g_rmse = node_errors(ucg.cpu().numpy(), N, sec41_exact)
        ref = PAPER_TABLE1.get(N)
        rows.append({"N": N, "h": f"2/{N}", "batch": batch, "steps": steps, "rmse": rmse,
                     "linf": linf, "s_per_epoch": wall / epochs,
                     "grid_cg": {"rmse": g_rmse, "linf": g_linf, "iterations": it_cg,
                                 "converged": ok_cg},
                     "final_loss": float(hist[:k].mean()),
                     "paper_rmse": ref[0] if ref else None, "paper_linf": ref[1] if ref else None,
                     "paper_s_per_epoch": ref[2] if ref else None})
    return {"metric": "Sec. 4.1 convergence study (Table 1 of the paper)", "epochs": epochs,
            "lr": lr, "networks": "2 x (3 -> 5 x 10 sine -> 1), 982 parameters, FP32",
            "rows": rows}


def cpu_baseline_grid():
    """The FP64 oracle's grid solve (row assembly and Jacobi PCG, OpenMP over
    rows, all host cores) on the grid_solves problem at 64^3 and 128^3 node
    grids, rtol 1e-10."""
    from oracle import pyoracle as O
    O.build()
    pr = O.make_problem(geometry=O.GEOM_SPHERE, mu_minus=1.0, mu_plus=10.0)
    out = {"kind": "oracle", "cores": O.default_threads()}
    for n in (64, 128):
        t0 = time.perf_counter()
        st, _, it, rr = O.grid_cg_solve(pr, n, rtol=1e-10, max_iter=100000)
        wall = time.perf_counter() - t0
        out[f"grid_cg_{n}"] = {"unknowns": (n - 1) ** 3, "iterations": it, "relres": rr,
                               "converged": st == 0, "wall_s": wall}
    return out


def grid_solves(hbm_peak, peak_src):
    """The grid scheme (sphere, mu 1/10) at 128^3 and 256^3 unknown grids to
    rtol 1e-10: FP64 Jacobi PCG and the refined solve (FP32 inner PCG on FP64
    residuals), with the exact node jump; and at 256^3 the refined solve with
    the extrapolated, lagged node jump."""
    import torch

    import paper_2210_14907_gb300 as nbm
    out = {}
    for n in (128, 256):
        dcg = nbm.ProblemDesc(geometry=nbm.GEOM_SPHERE, mu_minus=1.0, mu_plus=10.0)
        pcg = nbm.Problem(dcg)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        ucg, it, rr, ok = pcg.grid_cg_solve(n, rtol=1e-10, max_iter=100000)
        torch.cuda.synchronize()
        wall = time.perf_counter() - t0
        m = (n - 1) ** 3
        # algorithmic bytes per unknown and iteration of the streaming kernels (scaled
        # system): SpMV 40 + update 24 + direction 40.  128^3 runs from L2 and shared
        # memory in one cooperative kernel, so it has no HBM figure.
        gbs = it * 104 * m / wall / 1e9 if n > 130 else None
        linf, rmse = node_errors(ucg.cpu().numpy(), n)
        out[f"grid_cg_{n}"] = {"unknowns": m, "iterations": it, "relres": rr, "converged": ok,
                               "wall_s": wall, "achieved_gbs": gbs,
                               "hbm_frac": gbs and gbs / hbm_peak, "hbm_peak": f"{hbm_peak} GB/s {peak_src} copy",
                               "linf_exact": linf, "rmse_exact": rmse}
        del ucg
        torch.cuda.empty_cache()
        # the same system to the same FP64 residual test by FP32 inner corrections
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        uref, it, rr, ok = pcg.grid_solve_refined(n, rtol=1e-10, max_iter=100000)
        torch.cuda.synchronize()
        wall = time.perf_counter() - t0
        gbs = it * 43 * m / wall / 1e9 if n > 130 else None  # FP32: SpMV 9 + update 13 + direction 21 B
        linf, rmse = node_errors(uref.cpu().numpy(), n)
        out[f"grid_refined_{n}"] = {"unknowns": m, "inner_iterations": it, "relres": rr,
                                    "converged": ok, "wall_s": wall, "achieved_gbs": gbs,
                                    "hbm_frac": gbs and gbs / hbm_peak, "linf_exact": linf,
                                    "rmse_exact": rmse}
        del uref
        torch.cuda.empty_cache()
    dj = nbm.ProblemDesc(geometry=nbm.GEOM_SPHERE, mu_minus=1.0, mu_plus=10.0,
                         grid_jump=nbm.JUMP_EXTRAP)
    pj = nbm.Problem(dj)
    n, m = 256, 255 ** 3
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    uj, it, rr, ok = pj.grid_solve_refined(n, rtol=1e-10, max_iter=100000)
    torch.cuda.synchronize()
    wall = time.perf_counter() - t0
    passes, djump, fell_back = pj.grid_jump_info()
    linf, rmse = node_errors(uj.cpu().numpy(), n)
    out["grid_refined_256_lagged_jump"] = {"unknowns": m, "passes": passes, "fell_back": fell_back,
                                           "inner_iterations": it, "relres": rr, "converged": ok,
                                           "wall_s": wall, "linf_exact": linf, "rmse_exact": rmse}
    del uj
    torch.cuda.empty_cache()
    return out


def eval_grid_bench(dev, peak_src, tc_burst):
    """The surrogate on a dense 513^3 node grid (FP16 tcgen05 hidden layers, the
    flower-interface 3->128x4->1 architecture): grid points/s and its share of
    the burst 16-bit tensor peak, the best of three timed evaluations."""
    import torch

    import paper_2210_14907_gb300 as nbm
    d = nbm.config("C5")
    prob = nbm.Problem(d)
    params = nbm.xavier_init(d, seed=0, device=dev)
    n = 512
    nodes = (n + 1) ** 3
    u = torch.empty(nodes, device=dev)
    prob.eval_grid(params, n, precision=nbm.PREC_FP16, out=u)
    times = []
    for _ in range(3):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        prob.eval_grid(params, n, precision=nbm.PREC_FP16, out=u)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    ms = min(times)
    flops = nodes * 3 * 2 * 128 * 128  # hidden GEMMs of the node's own network
    del u
    torch.cuda.empty_cache()
    return {"metric": "grid points/s (trained-surrogate inference)", "value": nodes / ms * 1e3,
            "unit": "grid points/s", "grid": "513^3 nodes", "precision": "fp16",
            "ms": ms, "tensor_tflops": flops / ms / 1e9,
            "tensor_frac": flops / ms / 1e9 / tc_burst,
            "tensor_peak": f"{tc_burst} TFLOP/s {peak_src} dense 16-bit, burst (kernel timed alone)"}


def secondary(dev, hbm_peak, peak_src, tc_burst, tc_sustained):
    """Grid evaluation (a dense 513^3 node grid, FP16 tcgen05 hidden layers, the
    flower-interface 3->128x4->1 architecture), the mixed training step of the C3
    and C4 workloads, and the grid solve of the same discretization at 128^3 and
    256^3 (the plain method the NBM lifts off its grid): FP64 CG, and the
    refined solve with FP32 inner corrections to the same FP64 residual test."""
    import torch

    import paper_2210_14907_gb300 as nbm
    out = {"eval_grid": eval_grid_bench(dev, peak_src, tc_burst)}
    # the other training workloads: flower with 30 % band points (C3) and the
    # fine-resolution sphere with FP64 rows (C4), mixed path, full batches
    for name, steps in (("C3", 20), ("C4", 6)):
        dt = nbm.config(name)
        pt = nbm.Problem(dt)
        params = nbm.xavier_init(dt, seed=0, device=dev)
        m = torch.zeros_like(params)
        v = torch.zeros_like(params)
        B = nbm.BATCH[name]
        pt.train_steps(params, m, v, 0, 2, B, lr=1e-3, seed=1)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        pt.train_steps(params, m, v, 2, steps, B, lr=1e-3, seed=1)
        b.record()
        torch.cuda.synchronize()
        ms = a.elapsed_time(b) / steps
        flops = B * 21 * (dt.n_hidden - 1) * 2 * 128 * 128
        out[f"train_{name}"] = {"points_per_s": B / ms * 1e3, "ms_per_step": ms, "batch": B,
                                "tensor_tflops": flops / ms / 1e9,
                                "tensor_frac": flops / ms / 1e9 / tc_burst,
                                "tensor_frac_of_sustained": flops / ms / 1e9 / tc_sustained,
                                "steps": steps}
        del pt, params, m, v
        torch.cuda.empty_cache()
    out.update(grid_solves(hbm_peak, peak_src))
    return out


def exact_nodes_torch(n, k0, k1, geometry, dev, r0=0.5, amp=0.1, lt=5.0, lp=3.0):
    """The benchmark configurations' manufactured pair on the node planes k0..k1-1
    of the (n+1)^3 grid (FP64, device): u- = e^x cos y sin z where phi <= 0,
    u+ = x^2 + y^2 + z^2 elsewhere; phi of the sphere or the flower (theta the
    polar angle from +z, psi the azimuth)."""
    import torch
    g = -1.0 + torch.arange(n + 1, device=dev, dtype=torch.float64) * (2.0 / n)
    z, y, x = torch.meshgrid(g[k0:k1], g, g, indexing="ij")
    r = torch.sqrt(x * x + y * y + z * z)
    if geometry == "sphere":
        phi = r - r0
    else:
        theta = torch.atan2(torch.sqrt(x * x + y * y), z)
        psi = torch.atan2(y, x)
        phi = r - r0 - amp * torch.sin(lt * theta) * torch.cos(lp * psi)
    um = torch.exp(x) * torch.cos(y) * torch.sin(z)
    return torch.where(phi <= 0, um, x * x + y * y + z * z)


def grid_errors_gpu(u, n, geometry, stride=1):
    """L-infinity and RMS error of the node values u ((n+1)^3, x fastest, on the
    device) against the exact solution over the interior nodes; stride > 1 uses
    only the nodes of the coarser grid of spacing stride * 2/n.  Slab by slab."""
    import torch
    n1 = n + 1
    U = u.view(n1, n1, n1)
    linf, ss, cnt = 0.0, 0.0, 0
    ks = list(range(stride, n, stride))
    for c in range(0, len(ks), 16):
        kk = ks[c:c + 16]
        ex = torch.stack([exact_nodes_torch(n, k, k + 1, geometry, u.device)[0] for k in kk])
        e = (U[kk].to(torch.float64) - ex)[:, stride:n:stride, stride:n:stride]
        linf = max(linf, float(e.abs().max()))
        ss += float((e * e).sum())
        cnt += e.numel()
    return linf, (ss / cnt) ** 0.5


def _train(nbm, d, dev, steps, batch, lr=1e-3, seed=1, params=None, m=None, v=None, step0=0,
           chunk=500):
    """steps Adam steps of problem d from Xavier init (or the given state) in
    chunks; returns (problem, params, m, v, step, seconds, mean loss of the last
    chunk)."""
    import torch
    prob = nbm.Problem(d)
    if params is None:
        params = nbm.xavier_init(d, seed=0, device=dev)
        m = torch.zeros_like(params)
        v = torch.zeros_like(params)
    hist = torch.zeros(chunk, device=dev)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    st, done, last = step0, 0, 0
    while done < steps:
        k = min(chunk, steps - done)
        st = prob.train_steps(params, m, v, st, k, batch, lr=lr, seed=seed, loss_hist=hist[:k])
        done += k
        last = k
    torch.cuda.synchronize()
    return prob, params, m, v, st, time.perf_counter() - t0, float(hist[:last].mean())


def _grid(prob, n, solver, geometry):
    import torch
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    f = prob.grid_cg_solve if solver == "fp64_cg" else prob.grid_solve_refined
    u, it, rr, ok = f(n, rtol=1e-10, max_iter=200000)
    torch.cuda.synchronize()
    wall = time.perf_counter() - t0
    linf, rmse = grid_errors_gpu(u, n, geometry)
    return u, {"solver": solver, "n": n, "iterations": it, "relres": rr, "converged": ok,
               "wall_s": wall, "linf": linf, "rmse": rmse}


def study_c4(nbm, dev, steps):
    """Config 4: the sphere at h = 2/1024 (1024^3 effective resolution),
    4,194,304 points per step, 3 -> 128^4 -> 1, BF16 GEMMs with FP64 rows;
    steps Adam steps, then the exact-solution error at the 1025^3 nodes, beside
    the grid method on the same 1024^3 grid."""
    import torch
    d = nbm.config("C4")
    prob, params, m, v, st, wall, fl = _train(nbm, d, dev, steps, nbm.BATCH["C4"])
    u = prob.eval_grid(params, 1024, precision=nbm.PREC_FP32)
    linf, rmse = grid_errors_gpu(u, 1024, "sphere")
    out = {"steps": steps, "batch": nbm.BATCH["C4"], "train_s": wall, "final_loss": fl,
           "points_per_s": steps * nbm.BATCH["C4"] / wall,
           "surrogate": {"nodes": "1025^3 (interior)", "linf": linf, "rmse": rmse}}
    for s2 in (4, 8):  # the same surrogate at the nodes of the 256^3 and 128^3 grids
        out["surrogate"][f"linf_at_{1024 // s2}"], out["surrogate"][f"rmse_at_{1024 // s2}"] = \
            grid_errors_gpu(u, 1024, "sphere", stride=s2)
    del u
    torch.cuda.empty_cache()
    pg = nbm.Problem(nbm.ProblemDesc(geometry=nbm.GEOM_SPHERE, mu_minus=1.0, mu_plus=10.0))
    ug, out["grid_refined_1024"] = _grid(pg, 1024, "refined", "sphere")
    del ug, pg
    torch.cuda.empty_cache()
    return out


def study_c5(nbm, dev, steps):
    """Configs 3 and 5: train the flower problem (mu 1/100, h = 2/256, 1,048,576
    points per step with 30 % band points, 3 -> 128^4 -> 1) for `steps` Adam
    steps; judge that surrogate on the 513^3 nodes (FP16 tensor-core evaluation
    timed; FP32 evaluation for the errors) against the FP64 grid CG (rtol 1e-10)
    of the same discretization on the 128^3 and 256^3 grids, on exact-solution
    error and wall time."""
    import torch
    d = nbm.config("C3")
    prob, params, m, v, st, wall, fl = _train(nbm, d, dev, steps, nbm.BATCH["C3"])
    out = {"train": {"steps": steps, "batch": nbm.BATCH["C3"], "train_s": wall,
                     "final_loss": fl}}
    n = 512
    u16 = torch.empty((n + 1) ** 3, device=dev)
    prob.eval_grid(params, n, precision=nbm.PREC_FP16, out=u16)
    times = []
    for _ in range(3):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        prob.eval_grid(params, n, precision=nbm.PREC_FP16, out=u16)
        b.record()
        torch.cuda.synchronize()
        times.append(a.elapsed_time(b))
    l16, r16 = grid_errors_gpu(u16, n, "flower")
    del u16
    u = prob.eval_grid(params, n, precision=nbm.PREC_FP32)
    sur = {"nodes": "513^3", "eval_ms_fp16": min(times), "linf": None, "rmse": None,
           "linf_fp16_eval": l16, "rmse_fp16_eval": r16}
    sur["linf"], sur["rmse"] = grid_errors_gpu(u, n, "flower")
    for s2 in (2, 4):
        sur[f"linf_at_{n // s2}"], sur[f"rmse_at_{n // s2}"] = grid_errors_gpu(u, n, "flower", s2)
    out["surrogate"] = sur
    del u
    torch.cuda.empty_cache()
    pg = nbm.Problem(nbm.ProblemDesc(geometry=nbm.GEOM_FLOWER, mu_minus=1.0, mu_plus=100.0))
    for ng in (128, 256):
        ug, out[f"grid_cg_{ng}"] = _grid(pg, ng, "fp64_cg", "flower")
        del ug
    torch.cuda.empty_cache()
    return out


def study_per_h(nbm, dev, steps, ns):
    """Both methods at each h: the sphere (mu 1/10, 3 -> 128^3 -> 1, uniform
    points) and the flower (mu 1/100, 3 -> 128^4 -> 1, 30 % band points), each
    surrogate trained for `steps` Adam steps on 262,144 points per step at
    h = 2/n, errors at the (n+1)^3 nodes; the grid method on the same grid with
    the exact node jump and with its own extrapolated (lagged) jump."""
    import torch
    rows = []
    for geom, name in ((nbm.GEOM_SPHERE, "sphere"), (nbm.GEOM_FLOWER, "flower")):
        for n in ns:
            d = nbm.config("C2") if name == "sphere" else nbm.config("C3")
            d.h = 2.0 / n
            prob, params, m, v, st, wall, fl = _train(nbm, d, dev, steps, 262_144)
            u = prob.eval_grid(params, n, precision=nbm.PREC_FP32)
            sl, sr = grid_errors_gpu(u, n, name)
            del u
            row = {"geometry": name, "n": n, "h": f"2/{n}",
                   "surrogate": {"linf": sl, "rmse": sr, "train_s": wall, "final_loss": fl}}
            mu_p = 10.0 if name == "sphere" else 100.0
            for jm, jn in ((nbm.JUMP_EXACT, "grid_exact_jump"), (nbm.JUMP_EXTRAP, "grid_extrap_jump")):
                pg = nbm.Problem(nbm.ProblemDesc(geometry=geom, mu_minus=1.0, mu_plus=mu_p,
                                                 grid_jump=jm))
                ug, row[jn] = _grid(pg, n, "refined", name)
                row[jn]["passes"] = pg.grid_jump_info()[0]
                del ug, pg
            rows.append(row)
            print(json.dumps({"per_h_row": row}), flush=True)
            torch.cuda.empty_cache()
    return rows


def trilinear_torch(u, n, x, jump=None, side=None, node_side=None):
    """Trilinear interpolation of the node values u ((n+1)^3, x fastest) at the
    points x [m][3] (FP64, device).  With the node jump J = u+ - u- and the
    sides (0: minus, 1: plus) of the points and of the nodes, each corner value
    is first carried to the point's side (u_q + J_q for a minus node seen from
    the plus side, u_q - J_q the other way): the scheme's own extension of a
    side's solution across the interface."""
    import torch
    n1 = n + 1
    t = (x + 1.0) * (n / 2.0)
    i0 = torch.clamp(torch.floor(t).long(), 0, n - 1)
    f = t - i0
    out = torch.zeros(len(x), dtype=torch.float64, device=x.device)
    for dz in (0, 1):
        for dy in (0, 1):
            for dx in (0, 1):
                w = ((f[:, 0] if dx else 1 - f[:, 0]) * (f[:, 1] if dy else 1 - f[:, 1])
                     * (f[:, 2] if dz else 1 - f[:, 2]))
                idx = (i0[:, 0] + dx) + n1 * ((i0[:, 1] + dy) + n1 * (i0[:, 2] + dz))
                val = u[idx]
                if jump is not None:
                    sq = node_side[idx]
                    val = val + torch.where(sq == side, torch.zeros_like(val),
                                            torch.where(side == 1, jump[idx], -jump[idx]))
                out += w * val
    return out


def study_gain(nbm, dev, steps):
    """What the trained surrogate gains over the plain method near and away from
    the interface: the C2 sphere problem (h = 2/128), the surrogate after `steps`
    Adam steps against the grid solution at the same h, between nodes, by
    trilinear interpolation of the raw node values and by the scheme's
    jump-aware interpolation (each corner carried to the point's side with the
    node jump), with the exact jump and with the grid's own extrapolated jump."""
    import numpy as np
    import torch
    d = nbm.config("C2")
    prob, params, m, v, st, wall, fl = _train(nbm, d, dev, steps, 262_144)
    n = 128
    rng = np.random.default_rng(0)
    m_pts = 200_000
    dirs = rng.normal(size=(m_pts, 3))
    dirs /= np.linalg.norm(dirs, axis=1)[:, None]
    near = dirs * (0.5 + rng.uniform(-4.0 / n, 4.0 / n, m_pts))[:, None]  # within 2h of Gamma
    far = rng.uniform(-1, 1, size=(4 * m_pts, 3))
    far = far[np.abs(np.linalg.norm(far, axis=1) - 0.5) > 8.0 / n][:m_pts]  # beyond 4h
    g = -1.0 + torch.arange(n + 1, device=dev, dtype=torch.float64) * (2.0 / n)
    Z, Y, X = torch.meshgrid(g, g, g, indexing="ij")
    node_side = (torch.sqrt(X * X + Y * Y + Z * Z) - 0.5 > 0).reshape(-1).long()
    out = {"steps": steps, "train_s": wall, "h": "2/128"}
    grids = {}
    for jm, jn in ((nbm.JUMP_EXACT, "exact_jump"), (nbm.JUMP_EXTRAP, "extrap_jump")):
        pg = nbm.Problem(nbm.ProblemDesc(geometry=nbm.GEOM_SPHERE, mu_minus=1.0, mu_plus=10.0,
                                         grid_jump=jm))
        ug, _, _, _ = pg.grid_solve_refined(n, rtol=1e-10, max_iter=200000)
        grids[jn] = (ug, pg.grid_node_jump(n, jm, ug))
    for label, pts in (("near_interface", near), ("away_from_interface", far)):
        xt = torch.from_numpy(pts).to(dev)
        r = torch.sqrt((xt * xt).sum(1))
        side = (r - 0.5 > 0).long()
        ex = torch.where(side == 0, torch.exp(xt[:, 0]) * torch.cos(xt[:, 1]) * torch.sin(xt[:, 2]),
                         (xt * xt).sum(1))
        us = prob.eval_points(params, xt.float().contiguous()).double()
        res = {"points": len(pts)}

        def err(y):
            e = (y - ex).abs()
            return {"linf": float(e.max()), "rmse": float(torch.sqrt((e * e).mean()))}
        res["surrogate"] = err(us)
        ug, _ = grids["exact_jump"]
        res["grid_trilinear_raw"] = err(trilinear_torch(ug, n, xt))
        for jn, (ug, J) in grids.items():
            res[f"grid_jump_aware_{jn}"] = err(trilinear_torch(ug, n, xt, J, side, node_side))
        out[label] = res
    out["surrogate_bytes"] = params.numel() * 4
    out["grid_solution_bytes"] = (n + 1) ** 3 * 8
    return out


def study_long_c2(nbm, dev, schedule):
    """The C2 'same L-infinity' comparison at a lower error level than 2000
    constant-lr steps reach: the same coarse-to-fine schedule for the mixed
    (BF16) and the FP32 step, the state carried from stage to stage; each stage
    (cells of spacing 2/n, lr) runs its steps on 262,144 points; errors at the
    129^3 nodes after every stage."""
    out = {"schedule": [{"n": n, "steps": k, "lr": lr} for n, k, lr in schedule]}
    for prec, name in ((nbm.PREC_BF16, "mixed_bf16"), (nbm.PREC_FP32, "fp32")):
        params = m = v = None
        st, total, stages = 0, 0.0, []
        for n, k, lr in schedule:
            d = nbm.config("C2", precision=prec)
            d.h = 2.0 / n
            prob, params, m, v, st, wall, fl = _train(nbm, d, dev, k, 262_144, lr=lr,
                                                      params=params, m=m, v=v, step0=st)
            total += wall
            u = prob.eval_grid(params, 128, precision=nbm.PREC_FP32)
            linf, rmse = grid_errors_gpu(u, 128, "sphere")
            stages.append({"n": n, "steps": k, "lr": lr, "linf": linf, "rmse": rmse,
                           "final_loss": fl})
        out[name] = {"stages": stages, "train_s": total, "linf": stages[-1]["linf"],
                     "rmse": stages[-1]["rmse"]}
        print(json.dumps({"long_c2": {name: out[name]}}), flush=True)
    out["mixed_over_fp32_linf"] = out["mixed_bf16"]["linf"] / out["fp32"]["linf"]
    return out


def study(args):
    """The accuracy study of the learned part (configs 3-5): prints one JSON
    line per part as it finishes, then the whole study."""
    import torch

    import paper_2210_14907_gb300 as nbm
    torch.cuda.set_device(0)
    dev = torch.device("cuda", 0)
    parts = [p for p in args.study_parts.split(",") if p]
    out = {"metric": "exact-solution errors of the trained surrogate and of the grid method"}
    for part in parts:
        t0 = time.perf_counter()
        if part == "c4":
            r = study_c4(nbm, dev, args.study_c4_steps)
        elif part == "c5":
            r = study_c5(nbm, dev, args.study_c3_steps)
        elif part == "per_h":
            r = study_per_h(nbm, dev, args.study_per_h_steps,
                            [int(x) for x in args.study_per_h_n.split(",")])
        elif part == "gain":
            r = study_gain(nbm, dev, args.study_gain_steps)
        elif part == "long_c2":
            r = study_long_c2(nbm, dev, [(16, 2000, 1e-3), (32, 2000, 1e-3), (64, 2000, 1e-3),
                                         (128, 4000, 1e-3), (128, 2000, 1e-4)])
        else:
            raise ValueError(part)
        out[part] = r
        print(json.dumps({part: r, "part_s": time.perf_counter() - t0}), flush=True)
    print(json.dumps(out), flush=True)
    return 0


def run_reference(args):
    ws, rank, _ = _dist(gpu=False)
    if rank != 0:
        return
    cb = cpu_baseline(target_s=args.ref_seconds, steps=args.steps, warmup=args.warmup)
    # each timed step is one sub-batch of the workload's step: ms_per_step is
    # the measured time of that sub-batch step, so steps x ms_per_step is the
    # timed region; value (points/s) is comparable with the GPU arm's
    line = {"impl": "reference", "metric": METRIC, "value": cb["value"], "unit": UNIT,
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": cb["ms_per_step"], "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "batch": cb["sub_batch"],
                       "workload_batch": BATCH,
                       "sampling": f"each step: {cb['sub_batch']} of the {BATCH} points of "
                                   "that step's batch (the sub-batch the oracle finishes "
                                   "in the time budget)",
                       "reference": "FP64 CPU oracle (the paper publishes no code)"},
            "cpu_baseline": cb,
            "e2e": {"value": cb["value"], "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--fp32-steps", type=int, default=None)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--ref-seconds", type=float, default=60.0,
                    help="--impl reference: about this many seconds for the K timed steps")
    ap.add_argument("--no-secondary", action="store_true")
    ap.add_argument("--no-accuracy", action="store_true")
    ap.add_argument("--table1", action="store_true",
                    help="run the Sec. 4.1 convergence study instead of the benchmark")
    ap.add_argument("--table1-epochs", type=int, default=10000)
    ap.add_argument("--table1-n", default="8,16,32,64")
    ap.add_argument("--grid-only", action="store_true",
                    help="run only the grid solves (128^3, 256^3) and print their JSON")
    ap.add_argument("--eval-only", action="store_true",
                    help="run only the 513^3 grid evaluation and print its JSON")
    ap.add_argument("--study", action="store_true",
                    help="run the accuracy study of the learned part instead of the benchmark")
    ap.add_argument("--study-parts", default="gain,per_h,c5,c4,long_c2")
    ap.add_argument("--study-c4-steps", type=int, default=5000)
    ap.add_argument("--study-c3-steps", type=int, default=5000)
    ap.add_argument("--study-per-h-steps", type=int, default=2000)
    ap.add_argument("--study-per-h-n", default="32,64,128,256,512")
    ap.add_argument("--study-gain-steps", type=int, default=2000)
    args = ap.parse_args()
    args.warmup = max(3, args.warmup)
    if args.impl == "reference":
        return run_reference(args)
    if args.study:
        return study(args)
    if args.eval_only:
        import torch
        torch.cuda.set_device(0)
        burst, _, _, peak_src = _peaks()
        print(json.dumps(eval_grid_bench(torch.device("cuda", 0), peak_src, burst)))
        return 0
    if args.grid_only:
        import torch
        torch.cuda.set_device(0)
        _, _, hbm, peak_src = _peaks()
        out = grid_solves(hbm, peak_src)
        if not args.no_cpu_baseline:
            out["cpu_baseline_grid"] = cpu_baseline_grid()
        print(json.dumps(out))
        return 0
    if args.table1:
        import torch
        torch.cuda.set_device(0)
        out = table1(torch.device("cuda", 0), args.table1_epochs,
                     [int(v) for v in args.table1_n.split(",")])
        print(json.dumps(out))
        return 0

    import numpy as np
    import torch

    import paper_2210_14907_gb300 as nbm

    ws, rank, local = _dist()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    stream = torch.cuda.current_stream()
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    burst, sustained, hbm, peak_src = _peaks()

    from paper_2210_14907_gb300.data_parallel import DataParallelTrainer, torch_all_reduce

    def make_stepper(prob, params, m, v):
        """One training step per call.  One GPU: the fused nbm_train_steps.
        Several: this rank's shard of the ws x BATCH-point batch, NCCL
        all-reduce of gradient and loss, replicated Adam."""
        if ws == 1:
            state = {"t": 0}

            def one(pts=None, loss_hist=None):
                state["t"] = prob.train_steps(params, m, v, state["t"], 1, BATCH, seed=1,
                                              pts=pts, loss_hist=loss_hist)
            return one
        tr = DataParallelTrainer(prob, params, m, v, ws * BATCH, rank=rank, world=ws,
                                 all_reduce=torch_all_reduce(), seed=1)

        def one(pts=None, loss_hist=None):
            loss = tr.step(pts=pts)
            if loss_hist is not None:
                loss_hist.copy_(loss)
        return one

    def timed_run(prec, steps, warmup, profile):
        d = nbm.config("C2", precision=prec)
        prob = nbm.Problem(d)
        params = nbm.xavier_init(d, seed=0, device=dev)
        m = torch.zeros_like(params)
        v = torch.zeros_like(params)
        one = make_stepper(prob, params, m, v)
        for _ in range(warmup):
            one()
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
               for _ in range(steps)]
        torch.cuda.synchronize()
        _barrier(ws)
        torch.cuda.synchronize()
        if profile:
            prob.profile(True)
        t_wall = time.perf_counter()
        for k in range(steps):
            flush.zero_()
            evs[k][0].record(stream)
            one()
            evs[k][1].record(stream)
        torch.cuda.synchronize()
        t_wall = time.perf_counter() - t_wall
        _barrier(ws)
        ms = sum(a.elapsed_time(b) for a, b in evs)
        fused = prob.profile(False) if profile else (None, None)
        assert torch.isfinite(params).all()
        return ms, fused, t_wall, prob, one

    clk = Clocks(local)
    clk.start()
    time.sleep(0.3)
    clk.begin()
    ms, (fused_ms, fused_n), wall, prob, one = timed_run(nbm.PREC_BF16, args.steps, args.warmup,
                                                          True)
    clk.end()
    ms_max = _max_over_ranks(ws, ms)
    value = ws * args.steps * BATCH / (ms_max / 1e3)

    # plain FP32 path on the same workload (the comparison the metric asks for)
    k32 = args.fp32_steps if args.fp32_steps is not None else max(5, args.steps // 40)
    ms32, _, _, _, _ = timed_run(nbm.PREC_FP32, k32, 3, False)
    ms32 = _max_over_ranks(ws, ms32)
    value32 = ws * k32 * BATCH / (ms32 / 1e3)
    clk.stop()
    clocks = clk.summary()

    # end to end through the public API: per step, the step's collocation points
    # are copied from pinned host memory and the step's loss is read back.  The
    # copies run on their own stream into two device buffers, so that step k+1's
    # points cross while step k computes (each copy waits until the step that
    # last read its buffer has finished; each step waits for its own copy), and
    # the host reads step k's loss once step k+1 is enqueued, so the device does
    # not idle while the host checks it.
    k_e2e = max(10, args.steps // 20)
    rng = np.random.default_rng(rank)
    host = torch.from_numpy(
        (-1.0 + rng.integers(1, 2**23, size=(k_e2e, BATCH, 3)) * 2.0**-22).astype(np.float32)
    ).pin_memory()
    dbuf = [torch.empty(BATCH, 3, device=dev) for _ in range(2)]
    ldt = torch.float32 if ws == 1 else torch.float64  # loss_hist (fused) / all-reduced loss
    hist = torch.zeros(1, device=dev, dtype=ldt)
    hl = [torch.zeros(1, dtype=ldt).pin_memory() for _ in range(2)]
    cur = torch.cuda.current_stream()
    copy_stream = torch.cuda.Stream(device=dev)
    copied = [torch.cuda.Event() for _ in range(2)]
    used = [torch.cuda.Event() for _ in range(2)]
    read = [torch.cuda.Event() for _ in range(2)]

    def stage(k):
        b = k % 2
        copy_stream.wait_event(used[b])  # (an event never recorded: no wait)
        with torch.cuda.stream(copy_stream):
            dbuf[b].copy_(host[k], non_blocking=True)
        copied[b].record(copy_stream)

    def check(k):
        read[k % 2].synchronize()
        assert np.isfinite(hl[k % 2].item())

    def e2e_steps(n):
        stage(0)
        for k in range(n):
            if k + 1 < n:
                stage(k + 1)  # the next step's points cross while this step runs
            b = k % 2
            cur.wait_event(copied[b])
            one(pts=dbuf[b], loss_hist=hist)
            used[b].record(cur)
            hl[b].copy_(hist, non_blocking=True)  # this step's loss to the host
            read[b].record(cur)
            if k > 0:
                check(k - 1)  # the previous step's loss, while this step runs
        check(n - 1)

    e2e_steps(3)  # untimed: first touch of the pinned buffers and the copy path
    torch.cuda.synchronize()
    _barrier(ws)
    t0 = time.perf_counter()
    e2e_steps(k_e2e)
    e2e_s = _max_over_ranks(ws, time.perf_counter() - t0)
    e2e = {"value": ws * k_e2e * BATCH / e2e_s, "unit": UNIT,
           "h2d_bytes_per_step": BATCH * 3 * 4, "d2h_bytes_per_step": hl[0].element_size(),
           "steps": k_e2e,
           "pipelining": "inputs copied on a second stream while the previous step computes; "
                         "each step's loss read on the host while the next step computes",
           "l2": "not flushed: back-to-back steps, as a training loop runs (the device-timed "
                 "value flushes L2 before every step)"}

    # roofline of the fused tcgen05 kernel: algorithmic FLOPs = 7 stencil
    # evaluations x (forward + input-gradient + weight-gradient) x 2 H^2 per
    # hidden GEMM layer, per collocation point
    H, NG = 128, 2
    flops_pt = 21 * NG * 2 * H * H
    per_launch = flops_pt * BATCH
    t_launch = fused_ms / max(fused_n, 1) / 1e3
    achieved = per_launch / t_launch / 1e12
    sha = fused_sources_sha16()
    traffic_ok = sha == FUSED_TRAFFIC["sources_sha16"]
    # the fused kernel runs about a millisecond at a time inside a timed region of
    # a few seconds at most, so the burst peak (a GEMM timed alone) applies
    roof = {"bound": "tensor", "achieved": achieved, "peak": burst,
            "peak_kind": f"bf16 dense, {peak_src} burst (cuBLAS GEMM timed alone)",
            "unit": "TFLOP/s", "frac": achieved / burst,
            "frac_of_sustained": achieved / sustained,
            "kernel": "k_step_tc (fused forward+residual+backward)",
            "launch_ms": t_launch * 1e3, "flops_per_launch": per_launch,
            "traffic": FUSED_TRAFFIC["bytes"] if traffic_ok else None,
            "traffic_source": ("ncu dram__bytes_read.sum + dram__bytes_write.sum of one "
                               f"launch, kernel sources sha256 {sha}") if traffic_ok else
                              f"no capture of the current kernel sources (sha256 {sha})"}
    # the plain FP32 path against its FFMA peak, at the clock the run saw
    mhz = clocks.get("sm_mhz") or SM_MAX_MHZ
    ffma_peak = SMS * FP32_LANES * 2 * mhz * 1e6 / 1e12
    fp32_tflops = flops_pt * BATCH / (ms32 / k32 / 1e3) / 1e12

    if rank != 0:
        return
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_max / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "bf16", "data": "synthetic",
            "config": {"workload": WORKLOAD, "batch": BATCH * ws, "batch_per_gpu": BATCH,
                       "h": "2/128",
                       "l2": "flushed between timed steps (256 MiB write outside the events)",
                       "parallelism": (f"data parallel over {ws} GPUs: NCCL all-reduce of the "
                                       "gradient and loss, replicated Adam") if ws > 1
                                      else "1 GPU"},
            "fp32_path": {"value": value32, "unit": UNIT, "steps": k32,
                          "ms_per_step": ms32 / k32, "mixed_speedup": value / value32,
                          "ffma_tflops": fp32_tflops, "ffma_peak_tflops": ffma_peak,
                          "ffma_frac": fp32_tflops / ffma_peak,
                          "ffma_peak_kind": (f"{SMS} SMs x {FP32_LANES} FP32 lanes x 2 FLOP x "
                                             f"{mhz:.0f} MHz (median SM clock of the run)")},
            "roofline": roof, "e2e": e2e,
            "gpu_launches": (LAUNCHES_PER_STEP if ws == 1 else LAUNCHES_PER_DP_STEP)
                            * args.steps,
            "clocks": clocks, "wall_s": wall}
    if ws == 1 and not args.no_secondary:
        line["secondary"] = secondary(dev, hbm, peak_src, burst, sustained)
    if ws == 1 and not args.no_accuracy:
        line["accuracy"] = accuracy(dev)
    if ws == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline()
        if not args.no_secondary:
            line["cpu_baseline_grid"] = cpu_baseline_grid()
    print(json.dumps(line), flush=True)


if __name__ == "__main__":
    main()
