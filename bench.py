"""Benchmark of the matrix-free multivector product Y = A X on GB300.

One step = one fe_apply over the whole workload (gather, sum-factorised
contractions, quadrature-point operation, transposed contractions,
colour-ordered assembly).  Default workload: the 32^3-cell periodic box,
p = 6, n_q = 8, n_vec = 64 (7,077,888 DoFs), FP64, with FP32 measured beside
it.  Inputs (3.6 GB per block in FP64) are far larger than L2, so no flush is
needed between steps.

Prints ONE JSON line (rank 0).  Under torchrun each rank applies its own copy
of the workload on its own GPU (weak scaling, no collective on the data path).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
"""
from __future__ import annotations

import argparse
import hashlib
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

from paper_2208_07129_gb300 import inputs  # noqa: E402

METRIC = "FE A·X GDoF-vectors/s, FP64 vs mixed (rel err ≤1e-6), % roofline; PCG time"
UNIT = "GDoF-vectors/s"

# Roofline denominators.  HBM: measured copy bandwidth.  ALU-bound kernels: the
# pipe's unit count times the maximum SM clock (GB300: 152 SMs; per SM and clock
# 2 FP64 FMA lanes -- a DFMA microbenchmark measured 1.19 TFLOP/s -- and 128 FP32
# FMA lanes).
SMS = 152


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            return json.load(f), "measured"
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "bf16_tflops_sustained": 1700.0, "sm_max_mhz": 2070.0}, "fallback"


def alu_peak_tflops(dtype: str, sm_max_mhz: float) -> float:
    lanes = {"f64": 2, "f32": 128}[dtype]
    return SMS * lanes * 2 * sm_max_mhz * 1e6 / 1e12


def flops_per_cell_vec(np_: int, nq: int, box: bool = True) -> int:
    """Algorithmic flops per cell and vector: 2 flops per multiply-add of the six
    N / N^T passes and six D~ / D~^T passes (Sec. 2.2 complexity), plus the
    quadrature-point operation: 16 per point on trilinear cells (symmetric 3x3
    apply: 15, value: 1), 4 on axis-aligned boxes, whose metric is diagonal
    (three scalings and the value)."""
    return 4 * (np_ ** 3 * nq + np_ ** 2 * nq ** 2 + np_ * nq ** 3) + 12 * nq ** 4 + (4 if box else 16) * nq ** 3


def bytes_per_apply(w, elem: int, geo_elem: int = 0) -> int:
    """Algorithmic HBM bytes: X read once, Y written once (elem bytes each), the
    V coefficient per point and the per-point metric (6 values) on trilinear
    meshes (geo_elem bytes each; default elem)."""
    nq3 = w.nq ** 3
    geo = w.num_cells * nq3 * (geo_elem or elem) * (7 if w.perturb_seed is not None else 1)
    return w.num_dofs * w.n_vec * 2 * elem + geo


class ClockSampler:
    """nvidia-smi clock / throttle sampling during the timed region."""
    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.gpu = gpu_index
        self.proc = None
        # the raw samples go to FE_BENCH_OUT (default: the system temporary directory)
        out_dir = os.environ.get("FE_BENCH_OUT") or tempfile.gettempdir()
        self.path = os.path.join(out_dir, f"clocks_bench_{os.getpid()}.csv")

    def __enter__(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=self.f, stderr=subprocess.DEVNULL)
            time.sleep(0.3)
        except Exception:
            self.proc = None
        return self

    def __exit__(self, *a):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
            self.f.close()

    def summary(self, sm_max_default: float):
        if self.proc is None or not os.path.exists(self.path):
            return {"sm_mhz": None, "sm_max_mhz": sm_max_default, "reasons": ["unsampled"]}
        rows = []
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                rows.append((float(parts[1]), float(parts[2]), float(parts[3]), parts[5:9]))
            except ValueError:
                continue
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": sm_max_default, "reasons": ["unsampled"]}
        load = [r for r in rows if r[2] > 300.0] or rows
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[i] for r in load for i, v in enumerate(r[3]) if v.lower() == "active"})
        return {"sm_mhz": statistics.median(r[0] for r in load), "sm_max_mhz": max(r[1] for r in rows),
                "power_w_max": max(r[2] for r in rows), "samples": len(load), "reasons": reasons}


def dist_init():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        import torch
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    return world, rank, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x: float, world: int) -> float:
    """Max of a per-rank scalar (timings: the slowest rank defines the step)."""
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    dev = "cuda" if dist.get_backend() == "nccl" else "cpu"
    t = torch.tensor([x], dtype=torch.float64, device=dev)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def aggregate_throughput(units_per_rank: int, ms_per_step: float, world: int) -> float:
    """Whole-job throughput in G units/s: every rank processes its own copy of
    the workload (weak scaling), the step takes the slowest rank's time."""
    return units_per_rank * world / (ms_per_step * 1e-3) / 1e9


def traffic_for(kernel: str, source_files):
    """Per-launch DRAM bytes of `kernel` from the committed ncu summary, if the
    kernel's sources are unchanged since that capture (else None)."""
    p = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(p):
        return None
    data = json.load(open(p))
    ent = data.get(kernel)
    if not ent:
        return None
    h = hashlib.sha256()
    for f in source_files:
        h.update(open(os.path.join(ROOT, f), "rb").read())
    if ent.get("source_sha256") != h.hexdigest():
        return None
    return ent.get("dram_bytes_per_launch_full")


KERNEL_SOURCES = ["paper_2208_07129_gb300/csrc/" + f
                  for f in ("fe_box.cuh", "fe_cells.cuh", "fe_arith.cuh", "fe_dispatch.cuh", "fe_cell_kernel.cuh")]
FP64_KERNEL = "cell_apply_box_kernel<double,7,8>"


def box_operations_per_cell_vec(np_: int, nq: int) -> int:
    """Operations (one FP64 pipe slot each: add, multiply or multiply-add) the
    box-cell kernel executes per cell and vector, pass by pass (fe_box.cuh):
    even-odd contractions with N, the separable stiffness in its factors, and
    N^T."""
    hq, oq, hp, op = (nq + 1) // 2, nq // 2, (np_ + 1) // 2, np_ // 2
    n, nt, k = hq * hp + oq * op, hp * hq + op * oq, hq * hq - 1 + oq * oq   # k: L and d L^T of both halves
    point = 5 * oq + 2 * (nq & 1)
    return (np_ * np_ * (2 * op + n) + np_ * nq * (2 * op + n) + nq * nq * (2 * op + n + k + 4 * oq)
            + nq * nq * (k + 4 * oq) + nq * nq * (k + 2 * oq + point + nt + 2 * op)
            + (np_ * nq + np_ * np_) * (2 * oq + nt + 2 * op))


class OracleSample:
    """The FP64 oracle as it stands, on the host cores, on a bounded block of
    the workload: a contiguous block of rows of A (from the middle of the
    mesh) is assembled once into CSR by the oracle (its own quadrature, cell
    matrix rows and merge; timed and reported as assembly_s, not part of the
    rate), then every timed run is the oracle's OpenMP CSR x block product
    over that block with the workload's n_vec columns."""

    MAX_ROWS = 16384

    def __init__(self, w, assembly_budget_s: float = 6.0):
        from oracle import oracle as orc
        self.orc, self.w = orc, w
        self.mesh = orc.Mesh(w.nx, w.ny, w.nz, periodic=w.periodic, vertices=w.vertices())
        self.Vo = w.potential_at(orc.quad_points(self.mesh, w.p, w.nq))
        self.X = inputs.random_block(w.num_dofs, w.n_vec, w.x_dist, w.x_seed)
        # size the block by the assembly rate of a small probe
        probe = 8 * orc.num_threads()
        t0 = time.perf_counter()
        self._assemble(probe)
        rate = probe / max(time.perf_counter() - t0, 1e-6)
        n = int(min(self.MAX_ROWS, w.num_dofs, max(probe, rate * assembly_budget_s)))
        t0 = time.perf_counter()
        self._assemble(n)
        self.assembly_s = time.perf_counter() - t0
        self.n_rows = n
        self.nnz = int(self.B.nnz)
        self.spmm_s = None

    def _assemble(self, n: int):
        r0 = max(0, min(self.w.num_dofs - n, self.w.num_dofs // 2))
        self.r0 = r0
        self.B = self.orc.assemble_rows(self.mesh, self.w.p, self.w.nq, np.arange(r0, r0 + n), Vq=self.Vo,
                                        mu=self.w.mu)

    def run(self, reps: int = 1) -> float:
        t0 = time.perf_counter()
        for _ in range(reps):
            self.orc.spmm(self.B, self.X)
        dt = (time.perf_counter() - t0) / reps
        self.spmm_s = dt
        return dt

    def sized(self, budget_s: float) -> int:
        """Products per timed run so that one run takes about budget_s."""
        if self.spmm_s is None:
            self.run(1)
        return max(1, int(budget_s / max(self.spmm_s, 1e-6)))

    def seconds_per_apply(self) -> float:
        return self.spmm_s / self.n_rows * self.w.num_dofs

    def result(self, reps: int, dt: float) -> dict:
        w = self.w
        return {"value": self.n_rows * w.n_vec / dt / 1e9, "unit": UNIT, "cores": self.orc.num_threads(),
                "kind": "oracle", "assembly_s": self.assembly_s, "rows": self.n_rows, "nnz": self.nnz,
                "sample": f"rows {self.r0}..{self.r0 + self.n_rows - 1} of {w.num_dofs} of A ({w.name}; "
                          f"{self.nnz} nonzeros) assembled once into CSR by the oracle in {self.assembly_s:.1f} s "
                          f"(not timed), then the oracle's OpenMP CSR x {w.n_vec}-vector block product over that "
                          f"block, {reps} products, {dt * 1e3:.1f} ms each"}


def cpu_baseline(w, budget_s: float = 8.0):
    o = OracleSample(w)
    reps = o.sized(budget_s)
    return o.result(reps, o.run(reps))


def cpu_pcg_extrapolated(w, iterations: int, budget_s: float = 4.0) -> dict:
    """The oracle's time to solution for Jacobi-PCG on `w`, extrapolated: one
    full oracle apply (the CSR x block rate measured on an assembled row block,
    scaled to all rows) times the FP64 iteration count of the GPU solve.
    Assembly, vector updates and reductions are not counted, so the figure is
    a lower bound."""
    o = OracleSample(w)
    reps = o.sized(budget_s)
    dt = o.run(reps)
    s_apply = o.seconds_per_apply()
    return {"kind": "oracle", "cores": o.orc.num_threads(), "extrapolated": True,
            "seconds_per_apply": s_apply, "iterations": iterations, "seconds_extrapolated": s_apply * iterations,
            "assembly_s_block": o.assembly_s,
            "sample": f"CSR x {w.n_vec}-column product over {o.n_rows} assembled rows of {w.num_dofs} "
                      f"({reps} products, {dt * 1e3:.1f} ms each), scaled to all rows; assembly and vector "
                      f"updates not counted"}


def bench_config(w) -> dict:
    """The `config` object of both arms' JSON lines (same keys)."""
    return {"workload": w.name, "dofs": w.num_dofs, "cells": w.num_cells, "p": w.p, "n_q": w.nq,
            "n_vec": w.n_vec, "l2": "inputs larger than L2 (3.6 GB per FP64 block), no flush"}


def run_reference(args):
    """Reference arm: the FP64 oracle on the host cores (rank 0 only).  Its
    row block is assembled once before the warm-up; each step is the oracle's
    CSR x block product over that block of the 32^3 workload."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    w = inputs.WORKLOADS["c2"]
    o = OracleSample(w)
    reps = o.sized(max(1.0, 40.0 / max(1, args.warmup + args.steps)))
    for _ in range(args.warmup):
        o.run(reps)
    vals, dts = [], []
    for _ in range(args.steps):
        dt = o.run(reps)
        dts.append(dt)
        vals.append(o.n_rows * w.n_vec / dt / 1e9)
    v = statistics.median(vals)
    cb = o.result(reps, statistics.median(dts))
    cb["value"] = v
    print(json.dumps({"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus,
                      "steps": args.steps, "warmup": args.warmup, "ms_per_step": statistics.median(dts) * 1e3,
                      "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
                      "data": "synthetic", "config": bench_config(w),
                      "cpu_baseline": cb, "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0,
                                                  "d2h_bytes_per_step": 0}}), flush=True)


def time_mode(fe, torch, ctx, w, mode, steps, warmup, world):
    """Device-timed applies (CUDA events on the launching stream) and per-launch
    duration of the cell kernel; returns (ms_per_step, launches_per_step)."""
    fe.fe_set_mode(ctx, mode)
    X = torch.from_numpy(w.make_x()).to(device="cuda", dtype=fe.block_dtype(ctx))
    Y = torch.empty_like(X)
    stream = torch.cuda.current_stream()
    for _ in range(warmup):
        fe.fe_apply(ctx, X, Y)
    torch.cuda.synchronize()
    barrier(world)
    torch.cuda.synchronize()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(steps + 1)]
    ev[0].record(stream)
    for k in range(steps):
        fe.fe_apply(ctx, X, Y)
        ev[k + 1].record(stream)
    torch.cuda.synchronize()
    barrier(world)
    per = [ev[k].elapsed_time(ev[k + 1]) for k in range(steps)]
    total = ev[0].elapsed_time(ev[steps])
    ms = max_over_ranks(total / steps, world)
    return ms, per, X, Y


def solve_bench(fe, torch, cpu: bool = True, inner_modes=("fp32",)):
    """Time to relative residual 1e-8 (every column, checked with the FP64
    operator) for the block PCG solve of the 24^3, p=6, 128-column problem,
    every solve run to the end on all 128 columns: FP64 Jacobi-PCG with the
    FP64 operator, FP64 Jacobi-PCG with the double-float operator, mixed
    precision (inner Jacobi-PCG in each of `inner_modes`, FP64 refinement:
    FP32 CUDA-core products, TF32 and BF16 tensor-core products), and the
    learned preconditioner inside the mixed solve."""
    w = inputs.WORKLOADS["c5"]
    ctx = fe.setup_workload(w)
    out = {"workload": w.name, "rtol": 1e-8, "columns": w.n_vec}
    try:
        Bd = torch.from_numpy(w.make_rhs()).cuda()
        X = torch.zeros_like(Bd)

        def run(precond, inner):
            X.zero_()
            r = fe.fe_solve(ctx, Bd, X, rtol=1e-8, max_it=50000, precond=precond, inner_mode=inner)
            r.pop("rel_res")
            return r

        for m in inner_modes:
            out[f"mixed_{m}_jacobi"] = run("jacobi", m)
        r = out["mixed_fp32_jacobi"] if "mixed_fp32_jacobi" in out else out[f"mixed_{inner_modes[0]}_jacobi"]
        out["fp64_jacobi"] = run("jacobi", "fp64")
        out["df64_jacobi"] = run("jacobi", "df64")
        best = min(out[f"mixed_{m}_jacobi"]["seconds"] for m in inner_modes)
        out["speedup_mixed_vs_fp64"] = out["fp64_jacobi"]["seconds"] / best
        out["speedup_df64_vs_fp64"] = out["fp64_jacobi"]["seconds"] / out["df64_jacobi"]["seconds"]
        if cpu:
            out["cpu_oracle_fp64_jacobi"] = cpu_pcg_extrapolated(w, out["fp64_jacobi"]["iterations"])
        # learned cell-patch preconditioner: trained on this operator's own Jacobi-PCG
        # trajectories (8 random right-hand sides, snapshots every 32 iterations,
        # energy-norm objective, checkpoint picked on 4 held-out right-hand sides),
        # then used inside the mixed solve.  Five epochs: in six-epoch runs the
        # fifth epoch's network was the one whose held-out solve beat Jacobi
        info = fe.fe_precond_train(ctx, n_rhs=8, snapshots=16, snapshot_every=32, epochs=5, batch=2048, lr=3e-3,
                                   traj_rtol=1e-6, seed=3, objective="energy", n_val=4)
        rl = run("learned", "fp32")
        out["mixed_fp32_learned"] = rl
        out["training"] = info
        out["learned_vs_jacobi_iterations"] = rl["iterations"] / max(1, r["iterations"])
        out["speedup_learned_vs_fp64"] = out["fp64_jacobi"]["seconds"] / rl["seconds"]
    finally:
        fe.fe_destroy(ctx)
    return out


def chfsi_bench(fe, torch, fp32_switch: float = 1e-2) -> dict:
    """Chebyshev-filtered subspace iteration (Algorithm 6) on the scaled
    operator M^-1/2 A M^-1/2: the full solve of the 8^3 case in FP64 and in
    double-float (FP64 data, double-float scaled products) and in the mixed
    mode (FP32 rounds until the residual is below fp32_switch, double-float
    FP64 rounds to the end), and one double-float FP64 round (Lanczos bound,
    orthonormalisation and projection of the start block, one degree-67
    filter pass, orthonormalisation, projection) of the paper-size 17^3 case
    with 1280 vectors.  Start blocks: seeded standard normal, drawn on the device."""
    def start(w):
        g = torch.Generator(device="cuda")
        g.manual_seed(w.x_seed)
        return torch.randn(w.num_dofs, w.n_vec, device="cuda", dtype=torch.float64, generator=g)

    out = {}
    w = inputs.WORKLOADS["e0"]
    ctx = fe.setup_workload(w)
    try:
        for mode in ("fp64", "df64", "fp32"):
            # untimed: the first use of each dense library routine loads its kernels
            U = start(w)
            fe.fe_chfsi(ctx, U, n_wanted=w.extra["n_wanted"], degree=2, tol=w.extra["tol"], max_iter=1,
                        filter_mode=mode, fp32_switch=fp32_switch)
            del U
        ev = {}
        for mode, tag in (("fp64", "fp64"), ("df64", "df64"), ("fp32", "mixed")):
            U = start(w)
            r = fe.fe_chfsi(ctx, U, n_wanted=w.extra["n_wanted"], degree=w.extra["degree"], tol=w.extra["tol"],
                            max_iter=60, filter_mode=mode, fp32_switch=fp32_switch)
            ev[tag] = r.pop("eigenvalues")
            res = r.pop("residuals")
            r["lowest_eigenvalues"] = ev[tag][:3].tolist()
            r["max_wanted_residual"] = float(res[:w.extra["n_wanted"]].max())
            out["full_solve_" + tag] = r
            del U
        nw = w.extra["n_wanted"]
        out["full_solve_workload"] = w.name
        out["mixed_vs_fp64_max_rel_eigenvalue_diff"] = float(np.max(np.abs(ev["mixed"][:nw] - ev["fp64"][:nw]) /
                                                                np.abs(ev["fp64"][:nw])))
        out["df64_vs_fp64_max_rel_eigenvalue_diff"] = float(np.max(np.abs(ev["df64"][:nw] - ev["fp64"][:nw]) /
                                                               np.abs(ev["fp64"][:nw])))
        out["speedup_mixed_vs_fp64"] = out["full_solve_fp64"]["seconds"] / out["full_solve_mixed"]["seconds"]
        out["speedup_df64_vs_fp64"] = out["full_solve_fp64"]["seconds"] / out["full_solve_df64"]["seconds"]
    finally:
        fe.fe_destroy(ctx)
    torch.cuda.empty_cache()
    w = inputs.WORKLOADS["e1"]
    ctx = fe.setup_workload(w)
    try:
        U = start(w)
        r = fe.fe_chfsi(ctx, U, n_wanted=w.extra["n_wanted"], degree=w.extra["degree"], tol=w.extra["tol"],
                        max_iter=1, filter_mode="df64")
        r.pop("eigenvalues")
        r.pop("residuals")
        units = w.num_dofs * w.n_vec * w.extra["degree"]
        flops = flops_per_cell_vec(w.p + 1, w.nq, w.perturb_seed is None) * w.num_cells * w.n_vec * w.extra["degree"]
        ach = flops / r["seconds_filter"] / 1e12
        pk = alu_peak_tflops("f64", measured_peaks()[0].get("sm_max_mhz", 2070.0))
        r["filter_value"] = units / r["seconds_filter"] / 1e9
        r["filter_unit"] = UNIT
        r["filter_fp64_equivalent_tflops"] = ach
        r["filter_vs_dfma_roof"] = ach / pk
        r["filter_kernel"] = "cell_apply_box_kernel<ff,7,8> (double-float scaled product)"
        out["one_round_paper_size_df64"] = r
        out["one_round_workload"] = w.name
        del U
    finally:
        fe.fe_destroy(ctx)
    torch.cuda.empty_cache()
    return out


def small_case_bench(fe, torch, steps: int = 50) -> dict:
    """The 4^3 p=4 Dirichlet case with 8 vectors (314 KB of FP64 data, L2
    resident, latency-bound): microseconds per product, no roofline claim."""
    w = inputs.WORKLOADS["c1"]
    ctx = fe.setup_workload(w)
    out = {"workload": w.name}
    try:
        X = torch.from_numpy(w.make_x()).cuda()
        Y = torch.empty_like(X)
        for mode in ("fp64", "df64"):
            fe.fe_set_mode(ctx, mode)
            for _ in range(5):
                fe.fe_apply(ctx, X, Y)
            torch.cuda.synchronize()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(steps):
                fe.fe_apply(ctx, X, Y)
            b.record()
            torch.cuda.synchronize()
            out[mode + "_us_per_apply"] = a.elapsed_time(b) / steps * 1e3
        out["launches_per_apply"] = 2   # every cell, then the colour-ordered gather
    finally:
        fe.fe_destroy(ctx)
    return out


def refined_bench(fe, torch, steps: int = 3) -> dict:
    """The one-level refined mesh with hanging nodes (14^3 coarse cells, the
    central 8^3 split, p = 6, 64 vectors): time per constrained product
    (distribute, map cell kernels, condense) in FP64 and double-float."""
    w = inputs.WORKLOADS["h1"]
    ctx = fe.fe_setup_refined(w.nx, w.ny, w.nz, w.p, w.nq, w.extra["refine_lo"], w.extra["refine_hi"], mu=w.mu)
    out = {"workload": w.name, "dofs": fe.fe_num_dofs(ctx), "cells": fe.fe_num_cells(ctx),
           "hanging_nodes": fe.fe_num_slaves(ctx), "n_vec": w.n_vec}
    try:
        fe.fe_set_potential(ctx, w.potential_at(fe.fe_quadrature_points(ctx)))
        n = fe.fe_num_dofs(ctx)
        g = torch.Generator(device="cuda")
        g.manual_seed(w.x_seed)
        X = torch.randn(n, w.n_vec, device="cuda", dtype=torch.float64, generator=g)
        Y = torch.empty_like(X)
        for mode in ("fp64", "df64"):
            fe.fe_set_mode(ctx, mode)
            for _ in range(3):
                fe.fe_apply(ctx, X, Y)
            torch.cuda.synchronize()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(steps):
                fe.fe_apply(ctx, X, Y)
            b.record()
            torch.cuda.synchronize()
            ms = a.elapsed_time(b) / steps
            out[mode] = {"ms_per_apply": ms, "value": n * w.n_vec / (ms * 1e-3) / 1e9, "unit": UNIT}
        del X, Y
    finally:
        fe.fe_destroy(ctx)
    torch.cuda.empty_cache()
    return out


def distorted_bench(fe, torch, steps: int = 2, rows: int = 24):
    """The perturbed 16^3, p = 8, n_vec = 256 workload (trilinear cells,
    per-point metric): time per apply and relative error against the FP64
    oracle on sampled rows, for every arithmetic mode."""
    from oracle import oracle as orc
    w = inputs.WORKLOADS["c3"]
    ctx = fe.setup_workload(w)
    out = {"workload": w.name, "dofs": w.num_dofs, "n_vec": w.n_vec, "sampled_rows": rows}
    try:
        X64 = w.make_x()
        mesh = orc.Mesh(w.nx, w.ny, w.nz, periodic=w.periodic, vertices=w.vertices())
        Vo = w.potential_at(orc.quad_points(mesh, w.p, w.nq))
        ridx = np.sort(np.random.default_rng(3).integers(0, w.num_dofs, rows))
        rt = torch.from_numpy(ridx).cuda()
        for mode in ("fp64", "fp32", "tf32", "bf16", "tf32x3"):
            fe.fe_set_mode(ctx, mode)
            dt = torch.float64 if mode == "fp64" else torch.float32
            X = torch.from_numpy(X64).to(device="cuda", dtype=dt)
            Y = torch.empty_like(X)
            fe.fe_apply(ctx, X, Y)
            torch.cuda.synchronize()
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(steps):
                fe.fe_apply(ctx, X, Y)
            b.record()
            torch.cuda.synchronize()
            ms = a.elapsed_time(b) / steps
            Xr = X.double().cpu().numpy()
            ref = orc.apply_rows(mesh, w.p, w.nq, Xr, ridx, Vq=Vo, mu=w.mu)
            got = Y[rt].double().cpu().numpy()
            out[mode] = {"ms_per_apply": ms, "value": w.num_dofs * w.n_vec / (ms * 1e-3) / 1e9, "unit": UNIT,
                         "rel_err_vs_oracle": float(np.linalg.norm(got - ref) / np.linalg.norm(ref))}
            del X, Y, Xr
    finally:
        fe.fe_destroy(ctx)
    return out


def batch_bench(fe, torch, steps: int = 2):
    """The uneven batch: 24 periodic problems (n ~ U{4..24}, p ~ U{3..8},
    n_vec log-uniform in [8, 512]) in FP64, one persistent launch per apply
    replayed from a CUDA graph, against the same problems applied one after
    another with their own launches."""
    ws = inputs.batch_workloads()
    ctxs, Xs, Ys = [], [], []
    out = {"problems": len(ws), "mode": "fp64"}
    try:
        for w in ws:
            ctx = fe.setup_workload(w)
            ctxs.append(ctx)
            X = torch.from_numpy(w.make_x()).cuda()
            Xs.append(X)
            Ys.append(torch.empty_like(X))
        units = sum(w.num_dofs * w.n_vec for w in ws)
        flops = sum(flops_per_cell_vec(w.p + 1, w.nq, w.perturb_seed is None) * w.num_cells * w.n_vec for w in ws)
        b = fe.fe_batch_create(ctxs, [w.n_vec for w in ws], mode="fp64", autotune=True)
        try:
            st = fe.fe_batch_stats(b, len(ws))
            fe.fe_batch_apply(b, Xs, Ys)
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(steps):
                fe.fe_batch_apply(b, Xs, Ys)
            e1.record()
            torch.cuda.synchronize()
            ms_b = e0.elapsed_time(e1) / steps
            st2 = fe.fe_batch_stats(b, len(ws))
        finally:
            fe.fe_batch_destroy(b)
        Yr = [torch.empty_like(y) for y in Ys]
        # per-problem launches of the default (even-odd) kernel: the same cell body
        for c, X, Y in zip(ctxs, Xs, Yr):
            fe.fe_apply(c, X, Y)
        torch.cuda.synchronize()
        e0.record()
        for _ in range(steps):
            for c, X, Y in zip(ctxs, Xs, Yr):
                fe.fe_apply(c, X, Y)
        e1.record()
        torch.cuda.synchronize()
        ms_s = e0.elapsed_time(e1) / steps
        same = all(torch.equal(a, c) for a, c in zip(Ys, Yr))
        out.update({"dofs_x_vectors": units, "ms_per_batch_apply": ms_b, "value": units / (ms_b * 1e-3) / 1e9,
                    "unit": UNIT, "tflops": flops / (ms_b * 1e-3) / 1e12,
                    "ms_per_problem_launches": ms_s, "speedup_vs_per_problem_launches": ms_s / ms_b,
                    "bitwise_equal_to_per_problem": same, "device_status": st2["device_status"],
                    "work_items": st["work_items"], "phases": st["phases"], "grid": st["grid"],
                    "autotune_ms": st["autotune_ms"], "vectors_per_cta": st["vectors_per_cta"],
                    "cells_per_item": st["cells_per_item"],
                    "shapes": [[w.nx, w.p, w.n_vec] for w in ws]})
        # the same batch with double-float arithmetic (FP64 data), measured in
        # a process of its own: in this process, after the work above, the
        # capture of its graph fails (an open defect), while a fresh process
        # builds and runs it
        del Yr
        Xs.clear()
        Ys.clear()
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        out["df64"] = df64_batch_subprocess(ms_b)
    finally:
        for c in ctxs:
            fe.fe_destroy(c)
    return out


def df64_batch_child(fe, torch, steps: int = 2) -> dict:
    """The uneven batch of batch_bench with double-float arithmetic (FP64
    data), in a process of its own: one untimed and `steps` timed batch
    applies (CUDA graph), then the per-problem double-float launches for the
    bitwise comparison."""
    ws = inputs.batch_workloads()
    ctxs, Xs, Ys = [], [], []
    try:
        for w in ws:
            ctx = fe.setup_workload(w)
            ctxs.append(ctx)
            fe.fe_set_mode(ctx, "df64")
            X = torch.from_numpy(w.make_x()).cuda()
            Xs.append(X)
            Ys.append(torch.empty_like(X))
        units = sum(w.num_dofs * w.n_vec for w in ws)
        b = fe.fe_batch_create(ctxs, [w.n_vec for w in ws], mode="df64", autotune=True)
        try:
            fe.fe_batch_apply(b, Xs, Ys)
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(steps):
                fe.fe_batch_apply(b, Xs, Ys)
            e1.record()
            torch.cuda.synchronize()
            ms_d = e0.elapsed_time(e1) / steps
            st = fe.fe_batch_stats(b, len(ws))
        finally:
            fe.fe_batch_destroy(b)
        Yr = [torch.empty_like(y) for y in Ys]
        for c, X, Y in zip(ctxs, Xs, Yr):
            fe.fe_apply(c, X, Y)
        torch.cuda.synchronize()
        return {"ms_per_batch_apply": ms_d, "value": units / (ms_d * 1e-3) / 1e9, "unit": UNIT,
                "bitwise_equal_to_per_problem": all(torch.equal(a, c) for a, c in zip(Ys, Yr)),
                "device_status": st["device_status"], "vectors_per_cta": st["vectors_per_cta"],
                "process": "own (fresh) process"}
    finally:
        for c in ctxs:
            fe.fe_destroy(c)


def df64_batch_subprocess(ms_fp64_batch: float) -> dict:
    """Run df64_batch_child in a fresh process on the same GPU and return its
    result (or the error), with the speedup over the FP64 batch."""
    env = {k: v for k, v in os.environ.items()
           if k not in ("RANK", "WORLD_SIZE", "LOCAL_RANK", "LOCAL_WORLD_SIZE", "MASTER_ADDR", "MASTER_PORT")}
    try:
        r = subprocess.run([sys.executable, os.path.abspath(__file__), "--df64-batch-child"], capture_output=True,
                           text=True, timeout=900, env=env, cwd=ROOT)
        lines = [ln for ln in r.stdout.splitlines() if ln.startswith("{")]
        if r.returncode != 0 or not lines:
            tail = r.stderr.strip().splitlines()
            return {"error": f"child exited {r.returncode}: {tail[-1] if tail else 'no output'}"}
        d = json.loads(lines[-1])
        d["speedup_vs_fp64_batch"] = ms_fp64_batch / d["ms_per_batch_apply"]
        return d
    except Exception as ex:  # noqa: BLE001
        return {"error": f"{type(ex).__name__}: {ex}"}


def profile_precond(fe, torch, n: int = 12, n_vec: int = 128, reps: int = 3):
    """A small case of the learned-preconditioner inference kernel for
    hardware-counter captures: n^3 cells, p = 6, n_vec columns, seeded random
    weights; prints the mean time per application (CUDA events)."""
    w = inputs.Workload(f"{n}^3 p=6", n, n, n, False, 6, 8, n_vec, "normal", 5, "gauss", v_seed=15, v_amp=0.125,
                        v_shift=1.0)
    ctx = fe.setup_workload(w)
    try:
        fe.fe_precond_init(ctx, seed=1)
        R = torch.from_numpy(w.make_rhs()).float().cuda()
        Z = torch.empty_like(R)
        fe.fe_precond_apply(ctx, R, Z)
        torch.cuda.synchronize()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            fe.fe_precond_apply(ctx, R, Z)
        b.record()
        torch.cuda.synchronize()
        ms = a.elapsed_time(b) / reps
        print(json.dumps({"workload": w.name, "n_vec": n_vec, "ms_per_precond_apply": ms,
                          "gflops_mlp": 4 * 128 * (w.p + 1) ** 3 * w.num_cells * n_vec / (ms * 1e-3) / 1e9}))
    finally:
        fe.fe_destroy(ctx)


def profile_apply(fe, torch, n: int, mode: str, n_vec: int = 64, reps: int = 2):
    """A small case of one mode's cell kernel for hardware-counter captures:
    n^3 periodic cells, p = 6, n_q = 8, n_vec vectors (the 32^3 workload's
    shape), `reps` products after setup; prints the time per product."""
    w = inputs.Workload(f"{n}^3 periodic, p=6, n_q=8, n_vec={n_vec}", n, n, n, True, 6, 8, n_vec, "normal", 2,
                        "gauss", v_seed=12)
    ctx = fe.setup_workload(w)
    try:
        fe.fe_set_mode(ctx, mode)
        X = torch.from_numpy(w.make_x()).to(device="cuda", dtype=fe.block_dtype(ctx))
        Y = torch.empty_like(X)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            fe.fe_apply(ctx, X, Y)
        b.record()
        torch.cuda.synchronize()
        print(json.dumps({"workload": w.name, "mode": mode, "ms_per_apply": a.elapsed_time(b) / reps}), flush=True)
    finally:
        fe.fe_destroy(ctx)


def profile_solve(fe, torch, iterations: int, inner: str = "fp32"):
    """A short block-PCG run on the 24^3, p=6, 128-column problem (inner mode
    `inner` with FP64 refinement, capped at `iterations` inner iterations)
    for per-kernel launch lists."""
    w = inputs.WORKLOADS["c5"]
    ctx = fe.setup_workload(w)
    try:
        B = torch.from_numpy(w.make_rhs()).cuda()
        X = torch.zeros_like(B)
        r = fe.fe_solve(ctx, B, X, rtol=1e-8, max_it=iterations, precond="jacobi", inner_mode=inner)
        r.pop("rel_res", None)
        print(json.dumps({"workload": w.name, "inner": inner, **r}), flush=True)
    finally:
        fe.fe_destroy(ctx)


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="c2")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--modes", default="fp64,fp32")
    ap.add_argument("--no-solve", action="store_true")
    ap.add_argument("--no-batch", action="store_true")
    ap.add_argument("--no-distorted", action="store_true")
    ap.add_argument("--no-chfsi", action="store_true")
    ap.add_argument("--no-refined", action="store_true")
    ap.add_argument("--profile-precond", type=int, default=0, help="cells per direction of a preconditioner-only run")
    ap.add_argument("--profile-apply", type=int, default=0, help="cells per direction of a one-mode apply run "
                                                                  "(mode: the first of --modes)")
    ap.add_argument("--profile-solve", type=int, default=0, help="inner iterations of a short 24^3 PCG run")
    ap.add_argument("--df64-batch-child", action="store_true", help=argparse.SUPPRESS)
    args = ap.parse_args()
    if args.impl == "reference":
        run_reference(args)
        return
    if args.df64_batch_child:
        # the double-float batch in a process of its own (started by batch_bench on rank 0)
        import torch
        from paper_2208_07129_gb300 import fe
        fe.lib()
        print(json.dumps(df64_batch_child(fe, torch)), flush=True)
        return

    import torch
    world, rank, local = dist_init()
    torch.cuda.set_device(local)
    from paper_2208_07129_gb300 import build, fe
    if rank == 0:
        build.build()
    barrier(world)
    fe.lib()
    if args.profile_precond:
        profile_precond(fe, torch, n=args.profile_precond)
        return
    if args.profile_apply:
        profile_apply(fe, torch, args.profile_apply, args.modes.split(",")[0])
        return
    if args.profile_solve:
        profile_solve(fe, torch, args.profile_solve)
        return
    peaks, peak_src = measured_peaks()
    w = inputs.WORKLOADS[args.workload]
    ctx = fe.setup_workload(w)
    n_colors = 8 if (w.periodic is False or all(n % 2 == 0 for n in (w.nx, w.ny, w.nz))) else 27
    f_cell = flops_per_cell_vec(w.p + 1, w.nq, w.perturb_seed is None)
    flops = f_cell * w.num_cells * w.n_vec
    units = w.num_dofs * w.n_vec

    modes = {}
    want = args.modes.split(",")
    extra_modes = [m for m in ("df64", "tf32", "bf16", "bf16s", "tf32x3") if m in want or args.modes == "fp64,fp32"]
    with ClockSampler(local) as clk:
        ms64 = ms32 = float("nan")
        X64 = Y64 = X32 = Y32 = None
        if "fp64" in want:
            ms64, per64, X64, Y64 = time_mode(fe, torch, ctx, w, "fp64", args.steps, max(3, args.warmup), world)
        if "fp32" in want:
            ms32, per32, X32, Y32 = time_mode(fe, torch, ctx, w, "fp32", args.steps, max(3, args.warmup), world)
        ms_tc = {}
        for m in extra_modes:
            ms_tc[m], _, Xt, Yt = time_mode(fe, torch, ctx, w, m, args.steps, max(3, args.warmup), world)
            ms_tc[m + "_sample"] = (Xt, Yt)
    clocks = clk.summary(peaks.get("sm_max_mhz", 2070.0))
    if len(want) == 1:
        # profiling runs of a single mode print the timing and stop
        if rank == 0:
            print(json.dumps({"workload": w.name, "modes": want, "ms_per_step": {"fp64": ms64, "fp32": ms32}}), flush=True)
        fe.fe_destroy(ctx)
        return

    # end to end through the public host-buffer call: H2D of X, apply, D2H of Y
    fe.fe_set_mode(ctx, "fp64")
    Xh = X64.cpu().pin_memory()
    Yh = torch.empty_like(Xh).pin_memory()
    fe.fe_apply_host(ctx, Xh, Yh)
    torch.cuda.synchronize()
    barrier(world)
    t0 = time.perf_counter()
    e2e_steps = max(2, min(args.steps, 5))
    for _ in range(e2e_steps):
        fe.fe_apply_host(ctx, Xh, Yh)
    torch.cuda.synchronize()
    e2e_s = max_over_ranks((time.perf_counter() - t0) / e2e_steps, world)

    # accuracy of both modes on sampled rows against the FP64 oracle
    acc = {}
    if rank == 0 and not args.no_cpu:
        from oracle import oracle as orc
        mesh = orc.Mesh(w.nx, w.ny, w.nz, periodic=w.periodic, vertices=w.vertices())
        Vo = w.potential_at(orc.quad_points(mesh, w.p, w.nq))
        rows = np.sort(np.random.default_rng(1).integers(0, w.num_dofs, 48))
        ridx = torch.from_numpy(rows).cuda()
        pairs = [("fp64", X64, Y64), ("fp32", X32, Y32)] + [(m,) + ms_tc[m + "_sample"] for m in extra_modes]
        for mode, Xd, Yd in pairs:
            if Xd is None:
                continue
            Xr = Xd.double().cpu().numpy()
            Yref = orc.apply_rows(mesh, w.p, w.nq, Xr, rows, Vq=Vo, mu=w.mu)
            Yg = Yd[ridx].double().cpu().numpy()
            acc[mode] = float(np.linalg.norm(Yg - Yref) / np.linalg.norm(Yref))
            del Xr

    hbm = peaks["hbm_gbs"]
    sm_max = peaks.get("sm_max_mhz", 2070.0)
    total_units = units * world
    value = aggregate_throughput(units, ms64, world)
    value32 = aggregate_throughput(units, ms32, world)
    # dominant kernel: the cell kernel, n_colors launches per step; achieved =
    # algorithmic flops per launch / mean launch duration (event-timed step / launches)
    ach64 = flops / (ms64 * 1e-3) / 1e12
    exec64 = 2 * box_operations_per_cell_vec(w.p + 1, w.nq) * w.num_cells * w.n_vec / (ms64 * 1e-3) / 1e12
    if w.perturb_seed is not None:
        exec64 = ach64   # trilinear cells run the general kernel
    ach32 = flops / (ms32 * 1e-3) / 1e12
    pk64 = alu_peak_tflops("f64", sm_max)
    pk32 = alu_peak_tflops("f32", sm_max)
    b64 = bytes_per_apply(w, 8)
    b32 = bytes_per_apply(w, 4)
    traffic = traffic_for(FP64_KERNEL, KERNEL_SOURCES)
    modes["fp32"] = {
        "value": value32, "unit": UNIT, "ms_per_step": ms32, "dtype": "f32",
        "rel_err_vs_oracle": acc.get("fp32"),
        "roofline": {"bound": "alu", "achieved": ach32, "peak": pk32, "unit": "TFLOP/s", "frac": ach32 / pk32,
                     "hbm_frac": b32 / (ms32 * 1e-3) / 1e9 / hbm,
                     "peak_source": "152 SMs x 128 FP32 FMA/clk x 2 flop x max SM clock"},
    }
    for m in extra_modes:
        ach = flops / (ms_tc[m] * 1e-3) / 1e12
        if m == "df64":
            modes[m] = {"value": total_units / (ms_tc[m] * 1e-3) / 1e9, "unit": UNIT, "ms_per_step": ms_tc[m],
                        "dtype": "f64 data, double-float arithmetic (unevaluated pairs of f32) on the FP32 pipe",
                        "rel_err_vs_oracle": acc.get(m), "tolerance": 1e-12,
                        "fp64_equivalent_tflops": ach, "vs_dfma_roof": ach / pk64,
                        "speedup_vs_fp64": ms64 / ms_tc[m],
                        "hbm_frac": b64 / (ms_tc[m] * 1e-3) / 1e9 / hbm}
            continue
        io = 2 if m == "bf16s" else 4
        bt = bytes_per_apply(w, io, 4)
        gbs = bt / (ms_tc[m] * 1e-3) / 1e9
        modes[m] = {"value": total_units / (ms_tc[m] * 1e-3) / 1e9, "unit": UNIT, "ms_per_step": ms_tc[m],
                    "dtype": ("bf16 data, bf16 tensor-core contractions, f32 accumulation" if m == "bf16s" else
                              "f32 data, %s tensor-core contractions, f32 accumulation"
                              % ("split-TF32 (hi+lo, 3 products)" if m == "tf32x3" else m)),
                    "rel_err_vs_oracle": acc.get(m), "algorithmic_tflops": ach,
                    "kernel": "tc_apply_kernel (tcgen05)" if m != "tf32x3" else "mma_apply_kernel (warp MMA)",
                    "roofline": {"bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
                                 "algorithmic_bytes": bt},
                    "hbm_frac": gbs / hbm}
    out = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": max(3, args.warmup), "ms_per_step": ms64, "ms_per_step_median": statistics.median(per64),
        "ms_per_step_min": min(per64), "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": bench_config(w),
        "rel_err_vs_oracle": acc.get("fp64"), "sampled_rows": 48,
        "roofline": {"bound": "alu", "achieved": exec64, "peak": pk64, "unit": "TFLOP/s", "frac": exec64 / pk64,
                     "algorithmic_tflops": ach64, "traffic": traffic, "hbm_frac": b64 / (ms64 * 1e-3) / 1e9 / hbm,
                     "kernel": FP64_KERNEL,
                     "note": "achieved counts the FP64 operations the kernel executes, two flops per pipe slot; "
                             "algorithmic_tflops counts the sum-factorisation with D~ and D~^T, which the "
                             "separable stiffness of box cells undercuts",
                     "peak_source": f"152 SMs x 2 FP64 FMA/clk x 2 flop x {sm_max:.0f} MHz; HBM {hbm} GB/s {peak_src}"},
        "modes": modes,
        "e2e": {"value": total_units / e2e_s / 1e9, "unit": UNIT, "h2d_bytes_per_step": units * 8,
                "d2h_bytes_per_step": units * 8, "ms_per_step": e2e_s * 1e3,
                "path": "fe_apply_host with pinned host buffers: the FP64 cell kernels read X and write Y "
                        "in host memory over NVLink-C2C, no staging copies"},
        "gpu_launches": n_colors * args.steps,
        "clocks": clocks,
    }
    def section(fn, *a, **k):
        """One side section after the headline measurement: an error is
        recorded in its place, so the headline line is still printed."""
        try:
            return fn(*a, **k)
        except Exception as ex:  # noqa: BLE001
            return {"error": f"{type(ex).__name__}: {ex}"}

    if rank == 0 and not args.no_solve:
        out["pcg"] = section(solve_bench, fe, torch, cpu=not args.no_cpu, inner_modes=("fp32", "tf32", "bf16"))
    if rank == 0 and not args.no_batch:
        out["batch"] = section(batch_bench, fe, torch)
    if rank == 0 and not args.no_distorted:
        out["distorted"] = section(distorted_bench, fe, torch)
    if rank == 0 and not args.no_chfsi:
        out["chfsi"] = section(chfsi_bench, fe, torch)
    if rank == 0 and not args.no_refined:
        out["refined"] = section(refined_bench, fe, torch)
    if rank == 0:
        out["small_case"] = section(small_case_bench, fe, torch)
    if rank == 0 and not args.no_cpu:
        out["cpu_baseline"] = section(cpu_baseline, w)
    if rank == 0:
        print(json.dumps(out), flush=True)
    fe.fe_destroy(ctx)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
