#!/usr/bin/env python
"""Benchmark of the direct-solver hot path: Helmholtz RHS solves/s on one GB300.

Workload (one step): the k = 40 forward batch -- 32 x 32 leaves of 16 x 16
Chebyshev points on [-1, 1]^2, a smooth random contrast of 40 x 40 sine
coefficients (max |q| = 0.3), 128 plane waves and 256 receivers at R = 3.
A step factors the operator for that contrast (E_k, leaf operators, merges,
exterior coupling: hs_build), computes the total field of every incidence on
every leaf node (downward sweep) and the far field on the receivers
(hs_solve).  value = incidences solved per second, factorisation included.

Also reported: e2e (the same step through the host-buffer C-ABI calls, with
the host<->device copies inside the timed region), the FP64 roofline of the
dominant kernel family (the batched FP64 GEMM), the clocks seen during the
timed region, and the CPU oracle timed on a bounded slice of the workload.

Usage: python bench.py [--gpus N --steps K --warmup W --impl hs|reference]
For N > 1 launch with torchrun; every rank runs its own replica of the step
(weak scaling, no data-path collective) and rank 0 prints one JSON line.
"""
from __future__ import annotations

import argparse
import csv
import io
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

HERE = os.path.dirname(os.path.abspath(__file__))
if HERE not in sys.path:
    sys.path.insert(0, HERE)

import synth  # noqa: E402

METRIC = "Helmholtz RHS solves/s (factorisation included), k=40 forward batch"
UNIT = "solves/s"
# CPU-oracle slice: same leaf resolution (k h = 2.5) as the benchmark tree.
ORACLE_SAMPLE = dict(k=10.0, n_leaf=8, M=32, P=64)


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="hs", choices=["hs", "reference"])
    ap.add_argument("--precision", default="mixed", choices=["mixed", "fp64"])
    ap.add_argument("--prof-family", default="fp32", choices=["fp64", "fp32"],
                    help="kernel family timed for the line's roofline in the main arm: the SIMT FP32 GEMMs "
                         "(the largest family of the mixed step) or the FP64 GEMMs")
    ap.add_argument("--no-fp64-arm", action="store_true")
    ap.add_argument("--no-secondary", action="store_true")
    ap.add_argument("--workload", default="fwd_k40", choices=list(synth.WORKLOADS))
    ap.add_argument("--e2e-steps", type=int, default=3)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--case", default=None, choices=["gn_k40", "jacobian_16x16_s64", "lsqr_k40", "lsqr_mixed_k40",
                                                      "tc_shapes", "tc_2048", "jacobian_k40", "emulated_gemm_shapes",
                                                      "lu_1792", "mixed_k20", "paper_gn_k70"],
                    help="run one named workload once, untimed, and exit (a target for profilers)")
    ap.add_argument("--table2", type=float, default=0.0,
                    help="also run the paper's reconstruction plan (Sec. 4: k = 1:0.25:K, LSQR at 1e-3, "
                         "triangular modes, 5%% noise) up to this K and report it in the format of Table 2")
    ap.add_argument("--c5-sweep", action="store_true",
                    help="also run the paper-scale recursive linearization (k = 1:0.25:70, up to 19,600 unknowns, "
                         "128 x 128 leaves, 280 x 280 data) on mixed-precision contexts with LSQR on the tensor-core "
                         "Jacobian; about 15 minutes")
    ap.add_argument("--examples", action="store_true",
                    help="also run the paper's Examples 1 and 2 (analytic contrasts, k = 1..14.25 and 1..9, "
                         "its plan and LSQR, no noise) and report the L2 error of the reconstruction per k")
    ap.add_argument("--paper-gn", action="store_true",
                    help="also time one FP64 Gauss-Newton step at the paper-scale top frequency (k = 70, "
                         "19,600 coefficients, 280 x 280 data; about 3 minutes)")
    ap.add_argument("--table1-kmax", type=int, default=128,
                    help="top frequency of the paper's Table 1 forward benchmark (k = 1, 2, 4, .., this)")
    ap.add_argument("--sweep-kmax", type=float, default=10.0,
                    help="top frequency of the timed recursive-linearization sweep (40 = the full k = 1..40 plan)")
    return ap.parse_args()


def config_of(w, nranks, precision="fp64"):
    return {"workload": w.name, "precision": precision, "k": w.k, "leaves": f"{w.n_leaf_side}x{w.n_leaf_side}", "leaf_order": 16,
            "sine_modes": f"{w.S}x{w.S}", "incidences_per_gpu": w.M, "receivers": w.P, "R": w.R,
            "contrast": "smooth random sine series, max|q|=0.3, seed 2", "parallelism": f"replicas x{nranks}",
            "l2": "working set > L2 (factors ~1 GB, fields 0.5 GB per step)"}


def oracle_sample():
    """Time the CPU oracle (factor + solves + far field) on the bounded slice."""
    from oracle import forward as F
    s = ORACLE_SAMPLE
    c = synth.smooth_random_coeffs(10, seed=2, qmax=0.3)
    al, th = synth.directions(s["M"]), synth.receivers(s["P"])
    t0 = time.perf_counter()
    fw = F.forward_from_coeffs(c, s["k"], s["n_leaf"])
    fw.solve_plane(al, th)
    dt = time.perf_counter() - t0
    return s["M"] / dt, dt


def oracle_desc():
    s = ORACLE_SAMPLE
    return (f"CPU oracle (sparse-LU collocation, FP64) on the k={s['k']:g} slice with {s['n_leaf']}x{s['n_leaf']} "
            f"leaves (same k*h as the benchmark tree), {s['M']} plane waves, {s['P']} receivers; "
            f"factor + solves per step, solves/s = incidences / step time")


def oracle_slice_config(nranks):
    """config block of the oracle slice the reference arm actually runs (a bounded
    sample of the k = 40 forward workload: same leaf resolution k h = 2.5, same
    contrast generator, a 16x smaller tree and 4x fewer incidences)."""
    s = ORACLE_SAMPLE
    return {"workload": f"oracle_slice_fwd_k{s['k']:g}_{s['n_leaf']}x{s['n_leaf']}leaves_{s['M']}dirs_{s['P']}recv",
            "sample_of": synth.WORKLOADS["fwd_k40"].name, "precision": "fp64", "k": s["k"],
            "leaves": f"{s['n_leaf']}x{s['n_leaf']}", "leaf_order": 16, "sine_modes": "10x10",
            "incidences_per_gpu": s["M"], "receivers": s["P"], "R": 3.0,
            "contrast": "smooth random sine series, max|q|=0.3, seed 2", "parallelism": f"replicas x{nranks}"}


def blas_info():
    """BLAS library behind NumPy/SciPy and the number of threads it runs (the
    oracle's dense layer-potential products and LU use it; its sparse LU,
    SuperLU, runs on one thread)."""
    out = {"vendor": None, "version": None, "threads": None, "sparse_lu": "SuperLU (scipy.sparse.linalg.splu), 1 thread"}
    try:
        cfg = np.show_config(mode="dicts")["Build Dependencies"]["blas"]
        out["vendor"], out["version"] = cfg.get("name"), cfg.get("version")
    except Exception:  # noqa: BLE001 - reporting only
        pass
    try:
        import ctypes
        libs = sorted({ln.split()[-1] for ln in open("/proc/self/maps") if "openblas" in ln and ".so" in ln})
        for path in libs:
            lib_ = ctypes.CDLL(path)
            for name in ("scipy_openblas_get_num_threads64_", "scipy_openblas_get_num_threads",
                         "openblas_get_num_threads64_", "openblas_get_num_threads"):
                fn = getattr(lib_, name, None)
                if fn is not None:
                    fn.restype = ctypes.c_int
                    out["threads"] = int(fn())
                    break
            if out["threads"]:
                break
    except Exception:  # noqa: BLE001 - reporting only
        pass
    return out


def oracle_gn_step_k5():
    """The CPU oracle on the k = 5 Gauss-Newton workload in full (4 x 4 leaves, 10 x 10
    modes, 16 x 32 data): forward solve from c = 0, Jacobian by one Frechet solve per
    mode, normal equations with the same Tikhonov rule as the GPU step (lambda_rel
    1e-4).  Data from the oracle's forward map of the true contrast (untimed)."""
    from oracle import forward as F
    w = synth.WORKLOADS["gn_k5"]
    al, th = synth.directions(w.M), synth.receivers(w.P)
    data, _ = F.forward_from_function(synth.gaussian_bumps(1), w.k, w.n_leaf_side).solve_plane(al, th)
    t0 = time.perf_counter()
    fw = F.forward_from_coeffs(np.zeros((w.S, w.S)), w.k, w.n_leaf_side)
    Fc, _ = fw.solve_plane(al, th)
    J = fw.jacobian(al, th, w.S, w.S)
    A = (J.conj().T @ J).real
    F.gn_step(J, (data - Fc).ravel(), 1e-4 * np.trace(A) / A.shape[0])
    return time.perf_counter() - t0


def dist_init():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch
        import torch.distributed as dist
        backend = "nccl" if torch.cuda.is_available() else "gloo"
        dist.init_process_group(backend)
    return world, rank, local


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x, world):
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device="cuda" if torch.cuda.is_available() else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""

    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.f = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        try:
            self.p = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.QUERY}", "--format=csv,noheader,nounits",
                                       "-i", str(index), "-lms", "200"], stdout=self.f, stderr=subprocess.DEVNULL)
        except OSError:
            self.p = None

    def stop(self):
        if self.p is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.p.terminate()
        self.p.wait(timeout=10)
        self.f.seek(0)
        rows = [r for r in csv.reader(io.StringIO(self.f.read())) if len(r) >= 9]
        os.unlink(self.f.name)
        sm = [float(r[1]) for r in rows if r[1].strip().replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].strip().replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({n for r in rows for n, v in zip(names, r[5:9]) if v.strip() == "Active"})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "samples": len(rows), "reasons": reasons}


def run_reference(args, world, rank):
    if rank != 0:
        return
    for _ in range(args.warmup):
        oracle_sample()
    times = []
    for _ in range(args.steps):
        times.append(oracle_sample()[1])
    dt = sum(times) / len(times)
    v = ORACLE_SAMPLE["M"] / dt
    bl = blas_info()
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt * 1e3, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": oracle_slice_config(world),
            "cpu_baseline": {"value": v, "unit": UNIT, "cores": bl["threads"] or os.cpu_count(), "kind": "oracle",
                             "sample": oracle_desc(), "host_cpus": os.cpu_count(), "blas": bl},
            "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def time_arm(hs, torch, w, c, precision, args, world, local, prof_family, extra_family=None):
    """Warm up and time one precision arm of the step; returns its measurements.  prof_family is
    profiled over the timed steps (a family that leaves the captured graphs in place); with
    extra_family the returned profile comes from one more, untimed step of that family instead."""
    stream = torch.cuda.current_stream()
    solver = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, precision, device=local, stream=stream.cuda_stream)
    ctx = solver.ctx
    alphas = torch.tensor(synth.directions(w.M), device="cuda")
    thetas = torch.tensor(synth.receivers(w.P), device="cuda")
    ufar = torch.empty((w.M, w.P, 2), dtype=torch.float64, device="cuda")
    u = torch.empty((w.M, w.n_leaf_side ** 2, 256, 2), dtype=torch.float64, device="cuda")

    def step():
        hs.hs_build(ctx, c, w.k)
        hs.hs_forward_dev(ctx, alphas, thetas, ufar, u)

    for _ in range(max(args.warmup, 3)):
        step()
    torch.cuda.synchronize()
    clocks = Clocks(local)
    barrier(world)
    torch.cuda.synchronize()
    n0 = solver.launch_count()
    hs.hs_prof_start(prof_family)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        step()
    e1.record(stream)
    torch.cuda.synchronize()
    barrier(world)
    prof = hs.hs_prof_stop()
    launches = solver.launch_count() - n0
    clk = clocks.stop()
    ms = max_over_ranks(e0.elapsed_time(e1) / args.steps, world)
    # phase split (one extra, untimed pass)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
    ev[0].record(stream)
    hs.hs_build(ctx, c, w.k)
    ev[1].record(stream)
    hs.hs_forward_dev(ctx, alphas, thetas, ufar, u)
    ev[2].record(stream)
    torch.cuda.synchronize()
    phases = {"build_ms": ev[0].elapsed_time(ev[1]), "forward_ms": ev[1].elapsed_time(ev[2]),
              "cold_k_note": "median of 3 steps, each at a new k (k + 0.001 j): the build then also assembles the "
                             "boundary-integral matrices S, D of that k, which the steady-state steps reuse"}
    # solves/s of the sweep alone (factorisation excluded)
    phases["solves_per_s_excl_build"] = w.M / (phases["forward_ms"] * 1e-3)
    tc = None
    if precision == hs.HS_MIXED:
        it, upd, est = hs.hs_refine_stats(ctx)
        phases["refine_passes"] = it
        phases["last_rel_update"] = upd
        phases["est_rel_error"] = est
        # tensor-core GEMM family, one more untimed step with per-launch events
        hs.hs_prof_start(hs.HS_PROF_GEMM_TC)
        step()
        torch.cuda.synchronize()
        tc = hs.hs_prof_stop()
    if extra_family is not None:
        # a family whose per-launch events need launch-by-launch passes (the FP32
        # products run inside captured graphs otherwise): one more untimed step
        hs.hs_prof_start(extra_family)
        step()
        torch.cuda.synchronize()
        prof = hs.hs_prof_stop()
    # cold-frequency steps: each at a k not seen before, so the build also assembles
    # the layer-potential matrices S, D of that k (cached per k, so the timed steps
    # at a fixed k skip it); a mixed context then replays its factorisation graph
    # with the new k in device memory
    cold = []
    for j in range(3):
        kc = w.k + 1e-3 * (j + 1)
        ec = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        ec[0].record(stream)
        hs.hs_build(ctx, c, kc)
        hs.hs_forward_dev(ctx, alphas, thetas, ufar, u)
        ec[1].record(stream)
        torch.cuda.synchronize()
        cold.append(ec[0].elapsed_time(ec[1]))
    cold_ms = float(np.median(cold))
    phases["cold_k_step_ms"] = cold_ms
    step()  # back at the workload's k: ufar and u hold its fields again
    torch.cuda.synchronize()
    uf = ufar.cpu().numpy()
    return dict(solver=solver, ctx=ctx, ms=ms, launches=launches, prof=prof, tc=tc, clocks=clk, phases=phases,
                ufar=uf[..., 0] + 1j * uf[..., 1], u=u, alphas=alphas)


def combined_field(hs, torch, local, w, c, ufar_green):
    """The k = 40 forward step with combined-field exterior rows (bm_eta = 1) on a mixed context:
    steady-state and cold-k step times beside the Green-identity arm, the far-field difference
    between the two exterior forms at the workload's regular k, and the step at a Dirichlet
    eigenvalue of the square next to it, k = (pi/2) sqrt(650) = 40.05, where Green's rows leave
    the coupled system singular: refinement passes, and the combined rows' far field on mixed
    and FP64 contexts."""
    stream = torch.cuda.current_stream()
    al = torch.tensor(synth.directions(w.M), device="cuda")
    th = torch.tensor(synth.receivers(w.P), device="cuda")
    uf = torch.empty((w.M, w.P, 2), dtype=torch.float64, device="cuda")
    u = torch.empty((w.M, w.n_leaf_side ** 2, 256, 2), dtype=torch.float64, device="cuda")
    out = {"bm_eta": 1.0, "workload": w.name, "precision": "mixed"}

    def timed(ctx, k, reps):
        ts = []
        for _ in range(reps):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            e[0].record(stream)
            hs.hs_build(ctx, c, k)
            hs.hs_forward_dev(ctx, al, th, uf, u)
            e[1].record(stream)
            torch.cuda.synchronize()
            ts.append(e[0].elapsed_time(e[1]))
        return ts

    S = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, hs.HS_MIXED, device=local, stream=stream.cuda_stream, bm_eta=1.0)
    timed(S.ctx, w.k, 3)
    out["step_ms"] = float(np.median(timed(S.ctx, w.k, 5)))
    out["solves_per_s"] = w.M / (out["step_ms"] * 1e-3)
    out["cold_k_step_ms"] = float(np.median([timed(S.ctx, w.k + 1e-3 * (j + 1), 1)[0] for j in range(3)]))
    timed(S.ctx, w.k, 1)
    f = uf.cpu().numpy()
    f = f[..., 0] + 1j * f[..., 1]
    out["farfield_rel_diff_vs_green_rows"] = float(np.linalg.norm(f - ufar_green) / np.linalg.norm(ufar_green))
    keig = 0.5 * math.pi * math.sqrt(650.0)
    timed(S.ctx, keig, 1)
    it, _, est = hs.hs_refine_stats(S.ctx)
    fm = uf.cpu().numpy()
    S.close()
    S64 = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, hs.HS_FP64, device=local, stream=stream.cuda_stream, bm_eta=1.0)
    timed(S64.ctx, keig, 1)
    f64 = uf.cpu().numpy()
    S64.close()
    res = {"k": keig, "refine_passes": it, "est_rel_error": est,
           "mixed_vs_fp64_farfield_rel_err": float(np.linalg.norm(fm - f64) / np.linalg.norm(f64))}
    G = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, hs.HS_MIXED, device=local, stream=stream.cuda_stream)
    try:
        timed(G.ctx, keig, 1)
        it_g, upd_g, _ = hs.hs_refine_stats(G.ctx)
        res["green_rows"] = {"refine_passes": it_g, "last_rel_update": upd_g}
    except hs.HSError as e:
        it_g, upd_g, _ = hs.hs_refine_stats(G.ctx)
        res["green_rows"] = {"status": str(e).split(":")[0], "refine_passes": it_g, "last_rel_update": upd_g}
    G.close()
    out["at_dirichlet_eigenvalue"] = res
    return out


def run_hs(args, world, rank, local):
    import torch

    from paper_1608_06871_gb300.build import build
    if local == 0:
        build()
    barrier(world)
    import paper_1608_06871_gb300 as hs

    torch.cuda.set_device(local)
    # A dedicated (non-default) stream: the library launches on it and the CUDA
    # events are recorded on it, so they bracket exactly the library's work.
    stream = torch.cuda.Stream()
    torch.cuda.set_stream(stream)
    w = synth.WORKLOADS[args.workload]
    c = synth.smooth_random_coeffs(w.S, seed=2, qmax=0.3)
    peak = hs.hs_peak_fp64(local, 300.0)
    peak32 = hs.hs_peak_fp32(local, 300.0)
    prec = hs.HS_MIXED if args.precision == "mixed" else hs.HS_FP64
    main = time_arm(hs, torch, w, c, prec, args, world, local, hs.HS_PROF_GEMM_FP64,
                    None if args.prof_family == "fp64" else hs.HS_PROF_GEMM_FP32)
    other = None
    if prec == hs.HS_MIXED and not args.no_fp64_arm:
        other = time_arm(hs, torch, w, c, hs.HS_FP64, args, world, local, hs.HS_PROF_GEMM_FP64)
        other["solver"].close()
    value = world * w.M / (main["ms"] * 1e-3)

    # e2e: the same step through the C ABI with host buffers (pinned), copies inside the timed region
    ctx = main["ctx"]
    c_pin = torch.tensor(c, dtype=torch.float64).pin_memory()
    al_pin = torch.tensor(synth.directions(w.M)).pin_memory()
    th_pin = torch.tensor(synth.receivers(w.P)).pin_memory()
    out_pin = torch.empty((w.M, w.P, 2), dtype=torch.float64).pin_memory()
    c_np = c_pin.numpy()
    ufar_d = torch.empty((w.M, w.P, 2), dtype=torch.float64, device="cuda")

    def step_e2e():
        hs.hs_build(ctx, c_np, w.k)
        a_dev = al_pin.to("cuda", non_blocking=True)
        t_dev = th_pin.to("cuda", non_blocking=True)
        hs.hs_forward_dev(ctx, a_dev, t_dev, ufar_d, main["u"])
        out_pin.copy_(ufar_d, non_blocking=True)
        torch.cuda.current_stream().synchronize()

    step_e2e()
    barrier(world)
    t0 = time.perf_counter()
    for _ in range(args.e2e_steps):
        step_e2e()
    e2e_s = max_over_ranks((time.perf_counter() - t0) / args.e2e_steps, world)
    h2d = 8 * (w.S * w.S + w.M + w.P)
    d2h = 16 * w.M * w.P

    secondary = gn_and_gradient_times(hs, torch, local) if not args.no_secondary else None
    if secondary is not None:
        secondary["sweep_ms"] = sweep_time(hs, torch, local, k_max=args.sweep_kmax)
        secondary["sweep_mixed_lsqr_k40_ms"] = sweep_time(hs, torch, local, k_max=40.0, mixed_lsqr=True)
        secondary["sweep_mixed_lsqr_k10_vs_fp64"] = sweep_time(hs, torch, local, k_max=10.0, mixed_lsqr=True,
                                                               compare_fp64=True)
        secondary["paper_table1"] = paper_table1(hs, torch, local, k_max=args.table1_kmax)
        if prec == hs.HS_MIXED:
            secondary["combined_field_k40"] = combined_field(hs, torch, local, w, c, main["ufar"])
        if args.table2 > 0:
            secondary["paper_table2"] = paper_table2(hs, torch, local, args.table2)
        if args.c5_sweep:
            secondary["paper_scale_sweep"] = paper_scale_sweep(hs, torch, local)
        if args.examples:
            secondary["paper_examples"] = {f"example{e}": paper_example_run(hs, torch, local, e) for e in (1, 2)}
        if args.paper_gn:
            secondary["paper_scale_gn_step_k70"] = paper_scale_gn(hs, torch, local)

    cpu = None
    if rank == 0 and not args.no_cpu_baseline:
        v, dt = oracle_sample()
        bl = blas_info()
        cpu = {"value": v, "unit": UNIT, "cores": bl["threads"] or os.cpu_count(), "kind": "oracle",
               "sample": oracle_desc(), "seconds": dt, "host_cpus": os.cpu_count(), "blas": bl}
        gn_s = oracle_gn_step_k5()
        cpu["gn_step_k5"] = {"value": gn_s * 1e3, "unit": "ms", "workload": synth.WORKLOADS["gn_k5"].name,
                             "includes": "oracle forward + Frechet Jacobian (one solve per mode) + normal equations"}
        if secondary is not None:
            secondary["gn_step_ms"]["cpu_oracle_ms"] = gn_s * 1e3

    if rank == 0:
        gemm_ms, gemm_flops, gemm_n = main["prof"]
        achieved = gemm_flops / (gemm_ms * 1e-3) / 1e12 if gemm_ms > 0 else None
        fp64_fam = args.prof_family == "fp64"
        fam_peak = peak if fp64_fam else peak32
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
                "warmup": max(args.warmup, 3), "ms_per_step": main["ms"], "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None,
                "dtype": "c64 factors + f64 refinement" if prec == hs.HS_MIXED else "f64", "data": "synthetic",
                "config": config_of(w, world, args.precision),
                "e2e": {"value": world * w.M / e2e_s, "unit": UNIT, "h2d_bytes_per_step": h2d,
                        "d2h_bytes_per_step": d2h},
                "gpu_launches": main["launches"],
                "roofline": {"bound": "alu",
                             "kernel": "k_gemm<FP64> (batched FP64 GEMM family)" if fp64_fam
                             else "k_gemm32 / k_gemm_dot <FP32> (SIMT FP32 GEMM family: merges, sweeps, LU "
                                  "updates, leaf operators; the largest family of the mixed step)",
                             "achieved": achieved, "peak": fam_peak, "unit": "TFLOP/s",
                             "frac": (achieved / fam_peak) if (achieved and fam_peak) else None,
                             "peak_source": ("measured FP64 DFMA rate (hs_peak_fp64, this run)" if fp64_fam
                                             else "measured FP32 FFMA rate (hs_peak_fp32, this run)"),
                             "traffic": GEMM64_TRAFFIC if (fp64_fam and prec == hs.HS_MIXED) else None,
                             "traffic_note": GEMM64_TRAFFIC_NOTE if (fp64_fam and prec == hs.HS_MIXED) else
                             "a family of dozens of product shapes per step (the sweeps', merges', leaf and root "
                             "products): no single DRAM figure describes it",
                             "launches": gemm_n,
                             "kernel_ms_per_step": gemm_ms / (args.steps if fp64_fam else 1),
                             "algorithmic_tflop_per_step": gemm_flops / (args.steps if fp64_fam else 1) / 1e12,
                             "measured_over": "the timed steps" if fp64_fam else
                             "one extra, untimed step run launch by launch (per-launch CUDA events)"},
                "phases": main["phases"], "clocks": main["clocks"],
                "parity": {"fp64_vs_cpu_oracle": "1e-10 far field, 1e-9 fields and Jacobian, 1e-7 GN step, 1e-9 "
                                                 "gradient (tests/test_gpu_*.py) on trees the oracle factors (up to "
                                                 "16 x 16 leaves, k <= 20)",
                           "this_workload": "no CPU oracle at k = 40 on 32 x 32 leaves (a sparse LU of 2.6e5 "
                                            "unknowns with a dense 1792 block): pinned by q = 0 and a radial "
                                            "contrast against its separated-variables ODE reference (1e-8), "
                                            "mixed checked against the FP64 arm below"}}
        if other is not None:
            err = float(np.linalg.norm(main["ufar"] - other["ufar"]) / np.linalg.norm(other["ufar"]))
            f64 = (other["prof"][1] / (other["prof"][0] * 1e-3) / 1e12) if other["prof"][0] > 0 else None
            line["fp64_arm"] = {"value": world * w.M / (other["ms"] * 1e-3), "ms_per_step": other["ms"],
                                "phases": other["phases"], "gpu_launches": other["launches"],
                                "gemm_fp64_tflops": f64,
                                "roofline": {"bound": "alu", "kernel": "k_gemm<FP64> (batched FP64 GEMM family)",
                                             "achieved": f64, "peak": peak, "unit": "TFLOP/s",
                                             "frac": (f64 / peak) if (f64 and peak) else None,
                                             "peak_source": "measured FP64 DFMA rate (hs_peak_fp64, this run)",
                                             "kernel_ms_per_step": other["prof"][0] / args.steps}}
            line["mixed_vs_fp64_farfield_rel_err"] = err
            line["mixed_speedup_vs_fp64"] = other["ms"] / main["ms"]
        line["tensor_gemm"] = tensor_gemm_standalone(hs, torch)
        if main.get("tc") and main["tc"][0] > 0:
            tc_ms, tc_flops, tc_n = main["tc"]
            ach = tc_flops / (tc_ms * 1e-3) / 1e12
            line["tensor_gemm"]["in_step"] = {"achieved": ach, "launches": tc_n, "kernel_ms_per_step": tc_ms,
                                              "issued_tflops": 6 * ach,
                                              "frac_issued": 6 * ach / line["tensor_gemm"]["peak"]}
        else:
            line["tensor_gemm"]["in_step"] = None
        line["tensor_gemm"]["in_step_note"] = (
            "in the step the per-shape choice keeps the tensor cores only where they take less than half the "
            "SIMT time (the root product, the large trailing updates): their FP32 accumulation is coarser than "
            "SIMT FMA chains, and with a looser choice the k = 70 solve needs a fourth refinement pass")
        if secondary:
            line["secondary"] = secondary
        if cpu:
            line["cpu_baseline"] = cpu
        print(json.dumps(line), flush=True)
    main["solver"].close()


# DRAM bytes (read + write) of one launch of the dominant FP64 GEMM shape of the
# mixed step (the exterior-row residual [D - I/2, -S] [u_b; d_n u_b], 1792 x 128 x
# 3584 complex, two per step), from an ncu capture of the current kernel
# (dram__bytes_read.sum + dram__bytes_write.sum); its algorithmic bytes are
# 117.5 MB (the 1792 x 3584 matrix, the right-hand sides, C read and written).
GEMM64_TRAFFIC = None
GEMM64_TRAFFIC_NOTE = ("the mixed step's large FP64 products (exterior residual, far field) run on the emulated FP64 "
                       "product; the FP64 SIMT GEMMs left are small and their ncu traffic was taken on kernels that "
                       "have changed since")


def tensor_gemm_standalone(hs, torch):
    """The split-TF32 tensor-core product on 2048^3 and 4096^3 complex FP32 products (hs_gemm32 with
    the tensor cores forced; operand split kernels included), CUDA events, best of 3 after a
    warm-up; issued TF32 flops = 6 x useful (six split-term products)."""
    peak, src = tf32_peak()
    out = {"kernel": "k_t32_mma (tcgen05 kind::tf32, FP32 products by a three-term TF32 split, six products; "
                     "TMA 128B-swizzle ring, warp-specialised) + k_t32_split_rows / k_t32_split_cols",
           "bound": "tensor", "unit": "TFLOP/s", "peak": peak, "peak_source": src, "shapes": {}}
    g = torch.Generator(device="cuda").manual_seed(0)
    hs.hs_set_tensor_cores(2)
    try:
        for n in (2048, 4096):
            A = torch.complex(torch.randn((1, n, n), device="cuda", generator=g),
                              torch.randn((1, n, n), device="cuda", generator=g))
            B = torch.complex(torch.randn((1, n, n), device="cuda", generator=g),
                              torch.randn((1, n, n), device="cuda", generator=g))
            C = torch.empty_like(A)
            hs.hs_gemm32(A, B, C)
            torch.cuda.synchronize()
            best = 1e30
            for _ in range(3):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                hs.hs_gemm32(A, B, C)
                e1.record()
                torch.cuda.synchronize()
                best = min(best, e0.elapsed_time(e1))
            ach = 8.0 * n ** 3 / (best * 1e-3) / 1e12
            out["shapes"][f"{n}^3"] = {"ms": best, "achieved": ach, "issued_tflops": 6 * ach,
                                       "frac_issued": 6 * ach / peak}
            del A, B, C
    finally:
        hs.hs_set_tensor_cores(1)
    big = out["shapes"]["4096^3"]
    out.update(achieved=big["achieved"], frac_issued=big["frac_issued"])
    return out


def tf32_peak():
    """Dense TF32 tensor peak: the measured cuBLAS bf16 rate times the nominal
    TF32/BF16 ratio (1.1 / 2.25 PFLOP/s)."""
    try:
        with open(os.path.join(os.path.dirname(os.path.abspath(__file__)), "MEASURED_PEAKS.json")) as f:
            bf16 = float(json.load(f)["bf16_tflops"])
        return bf16 * 1.1 / 2.25, "measured bf16 burst (MEASURED_PEAKS.json) x nominal tf32/bf16 ratio 1.1/2.25"
    except (OSError, KeyError, ValueError):
        return 1900.0 * 1.1 / 2.25, "fallback bf16 1.9 PFLOP/s x nominal tf32/bf16 ratio 1.1/2.25"


def sweep_time(hs, torch, local, k_max=10.0, mixed_lsqr=False, compare_fp64=False):
    """Recursive-linearization sweep (Sec. 3.4): k = 1, 1.5, .., k_max with the
    ceil(1.6 k) modes / ceil(4 k) incidences and receivers / leaves-by-k plan,
    one Gauss-Newton step per frequency, blurred-ellipse phantom (seed 7) plus
    1% complex Gaussian noise.  FP64 with the direct normal equations, or
    (mixed_lsqr) on mixed-precision contexts with LSQR at 1e-3 on the
    FP32 Jacobian.  The data of every frequency are computed first on
    the GPU (untimed); the timed region is the whole sweep."""
    from paper_1608_06871_gb300 import sweep as SW
    plans = [SW.plan_ceil(float(k)) for k in np.arange(1.0, k_max + 0.25, 0.5)]
    phantom = synth.ellipse_phantom(7)
    data = {}
    for p in plans:
        al = 2 * np.pi * np.arange(p.M) / p.M
        th = 2 * np.pi * np.arange(p.P) / p.P
        gen = hs.Solver(p.leaves_per_side, 2, 2, 3.0, hs.HS_MIXED, device=local)
        x, y = gen.node_coords()
        gen.build_nodes(phantom(x, y), p.k)
        data[p.k] = synth.add_noise(gen.solve(al, th), 0.01, seed=70)
        gen.close()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    if mixed_lsqr:
        res = SW.recursive_linearization(plans, lambda p, al, th: data[p.k], device=local, precision=hs.HS_MIXED,
                                         solver="lsqr", lsqr_products=hs.HS_MIXED)
    else:
        res = SW.recursive_linearization(plans, lambda p, al, th: data[p.k], lambda_rel=1e-4, device=local)
    torch.cuda.synchronize()
    dt = time.perf_counter() - t0
    S = res.c.shape[0]
    c_true = synth.project_sine(phantom, S, S, nq=max(256, 4 * S))
    how = ("mixed precision, LSQR at 1e-3 on the FP32 Jacobian" if mixed_lsqr
           else "FP64, direct normal equations (lambda_rel 1e-4)")
    extra = {}
    if compare_fp64 and mixed_lsqr:
        # the same plan and data: (1) LSQR at 1e-3 on FP64 contexts (FP64 products), on mixed
        # contexts with FP64 products; (2) the direct Gauss-Newton step on FP64 and on mixed
        # contexts.  Each direct step is a continuous function of its inputs, so the mixed sweep
        # tracks the FP64 one to the refinement tolerance; LSQR stopped at a tolerance is not
        # (a perturbation at rounding level can move one frequency's stopping iteration by one,
        # which changes that step by about the tolerance and the rest of the sweep with it).
        def run(prec, solver):
            t1 = time.perf_counter()
            r = SW.recursive_linearization(plans, lambda p, al, th: data[p.k], device=local, precision=prec,
                                           solver=solver, lambda_rel=1e-4)
            return r, time.perf_counter() - t1
        r64, t64 = run(hs.HS_FP64, "lsqr")
        rmx, tmx = run(hs.HS_MIXED, "lsqr")
        d64, td64 = run(hs.HS_FP64, "direct")
        dmx, tdmx = run(hs.HS_MIXED, "direct")
        nrm, nrd = np.linalg.norm(r64.c), np.linalg.norm(d64.c)
        it64 = [h["lsqr_iterations"][0] for h in r64.history]
        itmx = [h["lsqr_iterations"][0] for h in rmx.history]
        extra = {"lsqr_fp64_sweep_ms": t64 * 1e3, "lsqr_mixed_fp64_products_sweep_ms": tmx * 1e3,
                 "lsqr_tensor_core_coeff_rel_diff_vs_fp64": float(np.linalg.norm(res.c - r64.c) / nrm),
                 "lsqr_mixed_fp64_products_coeff_rel_diff_vs_fp64": float(np.linalg.norm(rmx.c - r64.c) / nrm),
                 "lsqr_iteration_counts_that_differ": int(sum(a != b for a, b in zip(it64, itmx))),
                 "direct_fp64_sweep_ms": td64 * 1e3, "direct_mixed_sweep_ms": tdmx * 1e3,
                 "direct_mixed_coeff_rel_diff_vs_fp64": float(np.linalg.norm(dmx.c - d64.c) / nrd),
                 "note": "direct steps: the mixed sweep tracks the FP64 one to the refinement tolerance (the 1e-7 "
                         "coefficient bar); LSQR at 1e-3: differences of the order of the tolerance once one "
                         "frequency's stopping iteration moves"}
    return {"value": dt * 1e3, "unit": "ms", "frequencies": len(plans), **extra,
            "workload": f"sweep k=1:0.5:{k_max:g}, S=ceil(1.6k), M=P=ceil(4k), leaves 2^max(2,ceil(log2 0.8k)), "
                        f"ellipse phantom seed 7 + 1% noise, 1 GN step per k, {how}",
            "final_residual": float(res.history[-1]["residuals"][-1]),
            "coeff_rel_err_vs_phantom_projection": float(np.linalg.norm(res.c - c_true) / np.linalg.norm(c_true))}


def gn_and_gradient_times(hs, torch, local, reps=3):
    """GN-step time (k = 5 workload, FP64: build + solve + Jacobian + normal equations) and
    misfit-gradient time (k = 20 workload, FP64: build + forward + adjoint sweep), CUDA events."""
    stream = torch.cuda.current_stream()
    out = {}
    w = synth.WORKLOADS["gn_k5"]
    qt = synth.gaussian_bumps(1)
    al, th = synth.directions(w.M), synth.receivers(w.P)
    gen = hs.Solver(w.n_leaf_side, 2, 2, w.R, device=local, stream=stream.cuda_stream)
    x, y = gen.node_coords()
    gen.build_nodes(qt(x, y), w.k)
    data = gen.solve(al, th)  # measured data for the timing run (the parity test takes them from the oracle)
    gen.close()
    s = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, device=local, stream=stream.cuda_stream)
    c0 = np.zeros((w.S, w.S))
    ts = []
    for i in range(reps + 1):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        s.build(c0, w.k)
        s.gn_step(data, al, th, 1e-4, c0)
        e1.record(stream)
        torch.cuda.synchronize()
        if i:
            ts.append(e0.elapsed_time(e1))
    s.close()
    out["gn_step_ms"] = {"value": float(np.median(ts)), "workload": w.name, "precision": "fp64",
                         "includes": "hs_build + hs_gn_step (forward, Jacobian by adjoint sweep, normal equations)"}
    w = synth.WORKLOADS["grad_k20"]
    c = synth.project_sine(synth.ellipse_phantom(3), w.S, w.S)
    rng = np.random.default_rng(44)
    d = 0.05 * (rng.standard_normal((w.M, w.P)) + 1j * rng.standard_normal((w.M, w.P)))
    s = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, device=local, stream=stream.cuda_stream)
    ts = []
    for i in range(reps + 1):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        s.build(c, w.k)
        s.gradient(d, synth.directions(w.M), synth.receivers(w.P))
        e1.record(stream)
        torch.cuda.synchronize()
        if i:
            ts.append(e0.elapsed_time(e1))
    s.close()
    out["gradient_ms"] = {"value": float(np.median(ts)), "workload": w.name, "precision": "fp64",
                          "includes": "hs_build + hs_gradient (forward, adjoint sweep, projection)"}
    out["gn_step_k40"] = gn_step_top(hs, torch, local)
    out["paper_scale_forward_k70"] = paper_scale_forward(hs, torch, local)
    return out


def paper_scale_forward(hs, torch, local):
    """Forward batch at the top frequency of the paper-scale reconstruction:
    k = 70, 128 x 128 leaves (N = 3,690,241 distinct points), 140 x 140 = 19,600
    sine coefficients of a 40-inclusion contrast (seed 5, max|q| = 0.5), 280
    incidences to every leaf node plus the far field on 280 receivers; mixed
    precision and FP64, one warm-up and one timed build + forward each (CUDA
    events).  The paper's Table 1 row with the same N (12 cores, MATLAB):
    T_interior 1100 s, T_bdry 35.6 s, T_solve 87.1 ms per right-hand side."""
    stream = torch.cuda.current_stream()
    w = synth.WORKLOADS["fwd_k70"]
    c = synth.scaled_sine_coeffs(synth.inclusions(5), w.S, 0.5)
    alphas = torch.tensor(synth.directions(w.M), device="cuda")
    thetas = torch.tensor(synth.receivers(w.P), device="cuda")
    ufar = torch.empty((w.M, w.P, 2), dtype=torch.float64, device="cuda")
    u = torch.empty((w.M, w.n_leaf_side ** 2, 256, 2), dtype=torch.float64, device="cuda")
    out, far = {}, {}
    for name, prec in (("mixed", hs.HS_MIXED), ("fp64", hs.HS_FP64)):
        s = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, prec, device=local, stream=stream.cuda_stream)
        for _ in range(2):
            ev = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
            ev[0].record(stream)
            hs.hs_build(s.ctx, c, w.k)
            ev[1].record(stream)
            hs.hs_forward_dev(s.ctx, alphas, thetas, ufar, u)
            ev[2].record(stream)
            torch.cuda.synchronize()
        b_ms, f_ms = ev[0].elapsed_time(ev[1]), ev[1].elapsed_time(ev[2])
        out[name] = {"build_ms": b_ms, "forward_ms": f_ms, "solves_per_s": w.M / ((b_ms + f_ms) * 1e-3),
                     "solves_per_s_excl_build": w.M / (f_ms * 1e-3),
                     "forward_ms_per_rhs": f_ms / w.M}
        if prec == hs.HS_MIXED:
            it, upd, est = hs.hs_refine_stats(s.ctx)
            out[name].update(refine_passes=it, est_rel_error=est)
        uf = ufar.cpu().numpy()
        far[name] = uf[..., 0] + 1j * uf[..., 1]
        s.close()
    del u
    out["mixed_vs_fp64_farfield_rel_err"] = float(np.linalg.norm(far["mixed"] - far["fp64"]) /
                                                  np.linalg.norm(far["fp64"]))
    out["workload"] = w.name
    out["paper_table1_same_N"] = {"T_interior_s": 1100.0, "T_bdry_s": 35.6, "T_solve_s_per_rhs": 0.0871,
                                  "hardware": "MATLAB, up to 12 cores of a 2.5 GHz Xeon (context, not a target)"}
    return out


def paper_table2(hs, torch, local, k_max):
    """The paper's reconstruction plan (Sec. 4) with its solver: k = 1, 1.25, .., k_max;
    M = floor(2k) incidences, P = floor(4k) receivers at R = 20, unknowns the sine modes
    m1 + m2 <= floor(2k), one Gauss-Newton step per frequency with LSQR stopped at 1e-3,
    on [-pi/2, pi/2]^2 (computed on [-1, 1]^2 with k -> pi k / 2, R -> 2 R / pi).
    Contrast: the blurred-ellipse phantom (seed 7) standing in for the head phantom;
    data from the mixed-precision solver on a tree with twice the leaves per side
    (a different discretisation from the inversion's) plus 5% noise (seed 70).
    Reported like Table 2: N, Modes, M, M*P, T_f (factorisation), N_it (LSQR
    iterations), T_l (LSQR time), T_t (cumulative), in seconds."""
    from paper_1608_06871_gb300 import sweep as SW
    plans = [SW.plan_paper(float(k)) for k in np.arange(1.0, k_max + 1e-9, 0.25)]
    phantom = synth.ellipse_phantom(7)
    data = {}
    for p in plans:
        al = 2 * np.pi * np.arange(p.M) / p.M
        th = 2 * np.pi * np.arange(p.P) / p.P
        gen = hs.Solver(min(2 * p.leaves_per_side, 128), 2, 2, p.R, hs.HS_MIXED, device=local)
        x, y = gen.node_coords()
        data[p.k] = synth.add_noise(gen.build_nodes(phantom(x, y), p.k).solve(al, th), 0.05, seed=70)
        gen.close()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    res = SW.recursive_linearization(plans, lambda p, al, th: data[p.k], device=local, solver="lsqr")
    total = time.perf_counter() - t0
    rows, cum = [], 0.0
    for h in res.history:
        cum += h["t_f"][0] + h["t_l"][0]
        if float(h["k"]).is_integer() and (int(h["k"]) & (int(h["k"]) - 1)) == 0:
            rows.append({"k": h["k"], "N": h["N"], "Modes": h["modes"], "M": h["M"], "MP": h["M"] * h["P"],
                         "T_f": h["t_f"][0], "N_it": h["lsqr_iterations"][0], "T_l": h["t_l"][0], "T_t": cum})
    S = res.c.shape[0]
    c_true = synth.project_sine(phantom, S, S, nq=max(256, 4 * S)) * plans[-1].mask()
    return {"rows": rows, "frequencies": len(plans), "total_s": total,
            "coeff_rel_err_vs_phantom_projection": float(np.linalg.norm(res.c - c_true) / np.linalg.norm(c_true)),
            "note": "inverse on 4^l leaves with (pi k / 2) h <= 2.5 (finer than the paper's 6-10 points per "
                    "wavelength); paper's Table 2 (MATLAB, up to 32 cores): k = 16: T_f 2.99 s, N_it 27, "
                    "T_l 195.14 s, T_t 4109.56 s"}


# Table 1 of the paper (MATLAB, up to 12 cores of a 2.5 GHz Xeon): k -> (N, N_bdry, T_interior, T_bdry, T_solve)
PAPER_TABLE1 = {1: (3721, 640, 1.79, 1.94, 9.56e-4), 2: (3721, 640, 0.879, 1.70, 1.24e-3),
                4: (3721, 640, 0.857, 1.71, 1.74e-3), 8: (14641, 800, 4.12, 2.24, 1.47e-3),
                16: (58081, 1120, 16.6, 3.38, 2.95e-3), 32: (231361, 1760, 64.3, 5.96, 8.70e-3),
                64: (923521, 3040, 266.0, 12.3, 2.16e-2), 128: (3690241, 5600, 1100.0, 35.6, 8.71e-2)}


def paper_table1(hs, torch, local, k_max=128, M=64):
    """The paper's forward benchmark (Table 1) on its own workload: q = 1.5 exp(-|x|^2/50)
    (sign reading of synth.paper_example(1)) on [-pi/2, pi/2]^2, k = 1, 2, 4, ..., k_max,
    max(4, k)^2 leaves of 16 x 16 points (the table's N), M plane waves and M receivers.
    Per row and precision: T_interior and T_bdry of the first build at that k (CUDA events
    inside hs_build: leaves + merges; layer potentials + coupled root system + LU) and
    T_solve = time of hs_forward_dev for the M incidences (fields on every leaf node and
    the far field) / M.  The FP64 and mixed far fields are compared (relative L2)."""
    from paper_1608_06871_gb300 import sweep as SW
    stream = torch.cuda.current_stream()
    qfun = synth.paper_example(1)
    rows = []
    k = 1
    while k <= k_max:
        p = SW.plan_table1(float(k), M)
        al = torch.tensor(synth.directions(M), device="cuda")
        th = torch.tensor(synth.receivers(M), device="cuda")
        ufar = torch.empty((M, M, 2), dtype=torch.float64, device="cuda")
        u = torch.empty((M, p.leaves_per_side ** 2, 256, 2), dtype=torch.float64, device="cuda")
        row = {"k": k, "N": (15 * p.leaves_per_side + 1) ** 2, "N_bdry": 56 * p.leaves_per_side,
               "leaves": f"{p.leaves_per_side}x{p.leaves_per_side}"}
        far = {}
        for name, prec in (("fp64", hs.HS_FP64), ("mixed", hs.HS_MIXED)):
            if prec == hs.HS_MIXED:
                # a throwaway build first: the GEMM dispatch measures its FP32 product shapes once
                # per process, which must not land in the timed phases of the first build
                t = hs.Solver(p.leaves_per_side, 1, 1, p.R, prec, device=local, stream=stream.cuda_stream)
                tx, ty = t.node_coords()
                t.build_nodes(qfun(tx, ty), p.k)
                t.close()
            s = hs.Solver(p.leaves_per_side, 1, 1, p.R, prec, device=local, stream=stream.cuda_stream)
            x, y = s.node_coords()
            qn = qfun(x, y)
            s.build_nodes(qn, p.k)
            ti, tb = hs.hs_build_phase_ms(s.ctx)
            hs.hs_forward_dev(s.ctx, al, th, ufar, u)  # warm-up of the solve path
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            hs.hs_forward_dev(s.ctx, al, th, ufar, u)
            e1.record(stream)
            torch.cuda.synchronize()
            row[name] = {"T_interior_s": ti * 1e-3, "T_bdry_s": tb * 1e-3,
                         "T_solve_s_per_rhs": e0.elapsed_time(e1) * 1e-3 / M}
            if prec == hs.HS_MIXED:
                row[name]["refine_passes"] = hs.hs_refine_stats(s.ctx)[0]
            uf = ufar.cpu().numpy()
            far[name] = uf[..., 0] + 1j * uf[..., 1]
            s.close()
        del u
        row["mixed_vs_fp64_farfield_rel_err"] = float(np.linalg.norm(far["mixed"] - far["fp64"]) /
                                                      np.linalg.norm(far["fp64"]))
        pr = PAPER_TABLE1[k]
        row["paper"] = {"N": pr[0], "N_bdry": pr[1], "T_interior_s": pr[2], "T_bdry_s": pr[3],
                        "T_solve_s_per_rhs": pr[4]}
        rows.append(row)
        k *= 2
    return {"rows": rows, "rhs_per_solve": M,
            "note": "paper: MATLAB on up to 12 cores of a 2.5 GHz Xeon (context, not a target); its N_bdry is "
                    "its own exterior discretisation, here 56 n_L Chebyshev edge nodes"}


def paper_scale_sweep(hs, torch, local, k_max=70.0):
    """The paper-scale reconstruction: k = 1, 1.25, .., 70 (277 frequencies, plan_c5:
    S = floor(2k) modes per axis up to 140 x 140 = 19,600, M = P = ceil(4k) up to 280,
    leaves up to 128 x 128), one Gauss-Newton step per frequency by LSQR at 1e-3 on a
    mixed-precision context with the FP32 Jacobian.  Contrast: the 40-inclusion
    phantom (seed 5, max|q| = 0.5), data from the mixed solver on the same tree plus 1%
    noise (seed 70), generated before the timed sweep.  Reports rows at k = 1, 2, 4, ..,
    64, 70 like Table 2 (N, Modes, M*P, T_f, N_it, T_l, T_t) and the final coefficients'
    relative error against the contrast's projection on 140 x 140 modes."""
    from paper_1608_06871_gb300 import sweep as SW
    plans = [SW.plan_c5(float(k)) for k in np.arange(1.0, k_max + 1e-9, 0.25)]
    qfun = synth.inclusions(5)
    c_true = synth.scaled_sine_coeffs(qfun, int(math.floor(2 * k_max)), 0.5)
    scale = c_true[0, 0] / synth.project_sine(qfun, 1, 1, nq=640)[0, 0]
    data = {}
    t0 = time.perf_counter()
    for p in plans:
        al = 2 * np.pi * np.arange(p.M) / p.M
        th = 2 * np.pi * np.arange(p.P) / p.P
        gen = hs.Solver(p.leaves_per_side, 2, 2, p.R, hs.HS_MIXED, device=local)
        x, y = gen.node_coords()
        data[p.k] = synth.add_noise(gen.build_nodes(scale * qfun(x, y), p.k).solve(al, th), 0.01, seed=70)
        gen.close()
    t_data = time.perf_counter() - t0
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    res = SW.recursive_linearization(plans, lambda p, al, th: data[p.k], device=local, precision=hs.HS_MIXED,
                                     solver="lsqr", lsqr_products=hs.HS_MIXED)
    total = time.perf_counter() - t0
    rows, cum = [], 0.0
    for h in res.history:
        cum += h["t_f"][0] + h["t_l"][0]
        k = float(h["k"])
        if k == k_max or (k.is_integer() and (int(k) & (int(k) - 1)) == 0):
            rows.append({"k": k, "k_solver": h["k_solver"], "N": h["N"], "Modes": h["modes"], "MP": h["M"] * h["P"],
                         "T_f": h["t_f"][0], "N_it": h["lsqr_iterations"][0], "T_l": h["t_l"][0], "T_t": cum})
    return {"rows": rows, "frequencies": len(plans), "total_s": total, "data_generation_s": t_data,
            "coeff_rel_err_vs_contrast_projection": float(np.linalg.norm(res.c - c_true) / np.linalg.norm(c_true)),
            "paper_context": "~1e6 PDE solves in ~2 days of parallel MATLAB (Sec. 1, Sec. 4); Table 2: T_t = "
                             "151,114 s up to k = 64 for 8,128 modes"}


def paper_example_run(hs, torch, local, which):
    """The paper's Example 1 (k = 1..14.25) or 2 (k = 1..9), Sec. 4: its plan (k = 1 + j/4,
    M = floor(2k), P = floor(4k), R = 20, triangular modes, LSQR at 1e-3, one step per k)
    from the projection of q on the k = 1 modes, data without noise from the
    FP64 solver on a tree with twice the leaves per side.  Reports the L2 error
    of q_k on Omega (in the paper's units, over a 512^2 midpoint grid) at k = 1, 2, 3, ...
    and the total time (the paper: about 15 and 10 minutes on up to 32 cores)."""
    from paper_1608_06871_gb300 import sweep as SW
    qfun = synth.paper_example(which)
    k_top = 14.25 if which == 1 else 9.0
    plans = [SW.plan_paper(float(k)) for k in np.arange(1.0, k_top + 1e-9, 0.25)]
    data = {}
    for p in plans:
        al = 2 * np.pi * np.arange(p.M) / p.M
        th = 2 * np.pi * np.arange(p.P) / p.P
        gen = hs.Solver(min(2 * p.leaves_per_side, 128), 2, 2, p.R, device=local)
        x, y = gen.node_coords()
        data[p.k] = gen.build_nodes(qfun(x, y), p.k).solve(al, th)
        gen.close()
    c0 = synth.project_sine(qfun, plans[0].S, plans[0].S) * plans[0].mask()
    g = (np.arange(512) + 0.5) / 256.0 - 1.0
    X, Y = np.meshgrid(g, g, indexing="ij")
    q_ref = qfun(X, Y)
    cell = (math.pi / 512.0) ** 2  # area of a grid cell in the paper's units

    def l2_err(c):
        S = c.shape[0]
        bx = np.sin(np.outer(np.arange(1, S + 1), g + 1.0) * (math.pi / 2.0))
        return float(np.sqrt(np.sum((bx.T @ c @ bx - q_ref) ** 2) * cell))

    torch.cuda.synchronize()
    t0 = time.perf_counter()
    errs = []
    c = c0
    for j, p in enumerate(plans):  # one frequency at a time, to record the error after each
        res = SW.recursive_linearization([p], lambda pp, al, th: data[pp.k], c0=c, device=local, solver="lsqr")
        c = res.c
        if float(p.k_label).is_integer() or j == len(plans) - 1:
            errs.append({"k": p.k_label, "l2_err": l2_err(c), "lsqr_iterations": res.history[0]["lsqr_iterations"][0]})
    total = time.perf_counter() - t0
    best = synth.project_sine(qfun, plans[-1].S, plans[-1].S, nq=512) * plans[-1].mask()
    return {"l2_norm_q": float(np.sqrt(np.sum(q_ref ** 2) * cell)), "l2_error_by_k": errs, "total_s": total,
            "frequencies": len(plans), "initial_l2_err": l2_err(c0),
            "best_in_basis_l2_err": l2_err(best)}


def paper_scale_gn(hs, torch, local):
    """One Gauss-Newton step at the top frequency of the paper-scale reconstruction:
    k = 70, 128 x 128 leaves, 140 x 140 = 19,600 sine unknowns, 280 incidences x 280
    receivers (J: 78,400 x 19,600 complex).  Two ways, one timed run each (CUDA
    events): the paper's LSQR at 1e-3 on a mixed-precision context with the
    FP32 Jacobian (hs_build + hs_gn_step_lsqr), and the FP64 direct step
    (hs_build + hs_gn_step: Jacobian contraction, symmetric normal matrix, LU).
    Data: the 40-inclusion contrast (seed 5, max|q| = 0.5) plus 1% noise; the
    step starts from its first 120 x 120 coefficients."""
    stream = torch.cuda.current_stream()
    w = synth.WORKLOADS["fwd_k70"]
    c_true = synth.scaled_sine_coeffs(synth.inclusions(5), w.S, 0.5)
    al, th = synth.directions(w.M), synth.receivers(w.P)
    gen = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, hs.HS_MIXED, device=local, stream=stream.cuda_stream)
    data = synth.add_noise(gen.build(c_true, w.k).solve(al, th), 0.01, seed=70)
    gen.close()
    c = np.zeros_like(c_true)
    c[:120, :120] = c_true[:120, :120]
    out = {"workload": w.name, "unknowns": w.S * w.S, "jacobian_rows": w.M * w.P,
           "rel_err_before": float(np.linalg.norm(c - c_true) / np.linalg.norm(c_true)),
           "paper_context": "Table 2, k = 64 (8,128 modes, M*P = 65,536): T_f 25.97 s + LSQR T_l 1412.77 s on "
                            "up to 32 Xeon cores"}
    for name, prec in (("mixed_lsqr_tensor_core", hs.HS_MIXED), ("fp64_direct", hs.HS_FP64)):
        s = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, prec, device=local, stream=stream.cuda_stream)
        e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        e0.record(stream)
        s.build(c, w.k)
        e1.record(stream)
        if prec == hs.HS_MIXED:
            c1, rn, it = s.gn_step_lsqr(data, al, th, c, tol=1e-3, max_iter=500, products=hs.HS_MIXED)
        else:
            (c1, rn), it = s.gn_step(data, al, th, 1e-4, c), None
        e2.record(stream)
        torch.cuda.synchronize()
        s.close()
        out[name] = {"ms": e0.elapsed_time(e2), "build_ms": e0.elapsed_time(e1), "step_ms": e1.elapsed_time(e2),
                     "lsqr_iterations": it, "residual_norm": float(rn),
                     "rel_err_after": float(np.linalg.norm(c1 - c_true) / np.linalg.norm(c_true))}
    out["value"] = out["mixed_lsqr_tensor_core"]["ms"]
    out["unit"] = "ms"
    return out


def gn_step_top(hs, torch, local):
    """One Gauss-Newton step at the top frequency of the k = 1..40 sweep (k = 40,
    32 x 32 leaves, 64 x 64 = 4096 sine modes, 160 incidences, 160 receivers;
    blurred-ellipse phantom seed 7 with 1% noise as data, step from its
    projection on 40 x 40 modes), FP64: hs_build + hs_gn_step, CUDA events.
    Also times hs_jacobian_dev alone with the FP64 GEMM family's per-launch
    events (the contraction and the adjoint sweep's products)."""
    stream = torch.cuda.current_stream()
    w = synth.WORKLOADS["gn_k40"]
    phantom = synth.ellipse_phantom(7)
    al, th = synth.directions(w.M), synth.receivers(w.P)
    gen = hs.Solver(w.n_leaf_side, 2, 2, w.R, device=local, stream=stream.cuda_stream)
    x, y = gen.node_coords()
    gen.build_nodes(phantom(x, y), w.k)
    data = synth.add_noise(gen.solve(al, th), 0.01, seed=70)
    gen.close()
    c = np.zeros((w.S, w.S))
    c[:40, :40] = synth.project_sine(phantom, 40, 40)
    s = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, device=local, stream=stream.cuda_stream)

    ts = []
    for i in range(3):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        s.build(c, w.k)
        c1, rn = s.gn_step(data, al, th, 1e-4, c)
        e1.record(stream)
        torch.cuda.synchronize()
        if i:
            ts.append(e0.elapsed_time(e1))
    sm = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, hs.HS_MIXED, device=local, stream=stream.cuda_stream)
    # the direct step on a mixed context: FP32 factors, refined forward and adjoint fields,
    # FP64 contraction and normal equations
    ts_m = []
    for i in range(3):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        sm.build(c, w.k)
        c1m, rnm = sm.gn_step(data, al, th, 1e-4, c)
        e1.record(stream)
        torch.cuda.synchronize()
        if i:
            ts_m.append(e0.elapsed_time(e1))
    adj = hs.hs_adjoint_refine_stats(sm.ctx)
    mixed_direct = {"ms": float(np.median(ts_m)),
                    "step_rel_diff_vs_fp64": float(np.linalg.norm(c1m - c1) / np.linalg.norm(c1 - c)),
                    "adjoint_refine_passes": adj[0], "adjoint_est_rel_error": adj[2],
                    "includes": "hs_build + hs_gn_step on a mixed context (FP32 factors; forward and adjoint "
                                "fields refined in FP64; FP64 contraction and normal equations)"}
    variants = (("fp64_products", s, hs.HS_FP64), ("fp32_jacobian", s, hs.HS_MIXED),
                ("mixed_factors_fp64_products", sm, hs.HS_FP64),
                ("mixed_factors_fp32_jacobian", sm, hs.HS_MIXED))
    lsqr_out = {"tolerance": 1e-3,
                "includes": "hs_build + hs_gn_step_lsqr: forward, adjoint sweep, LSQR; fp64_products = J and J^H "
                            "applied from the fields in FP64 every iteration; fp32_jacobian = J formed once "
                            "in complex FP32 (the Khatri-Rao rows and two SIMT FP32 projections), LSQR products read it with FP64 sums; "
                            "mixed_factors = FP32 factors with forward and adjoint fields refined in FP64",
                "step_rel_diff_vs_fp64_at": "20 iterations each (tol 0)"}
    steps20 = {}
    for name, solver, prod in variants:
        ts_l = []
        for i in range(3 if name != "fp64_products" else 2):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record(stream)
            solver.build(c, w.k)
            _, _, it = solver.gn_step_lsqr(data, al, th, c, tol=1e-3, max_iter=500, products=prod)
            e1.record(stream)
            torch.cuda.synchronize()
            if i:
                ts_l.append(e0.elapsed_time(e1))
        solver.build(c, w.k)
        steps20[name] = solver.gn_step_lsqr(data, al, th, c, tol=0.0, max_iter=20, products=prod)[0] - c
        lsqr_out[name] = {"ms": float(np.median(ts_l)), "iterations": it}
    sm.close()
    for name, _, _ in variants[1:]:
        lsqr_out[name]["step_rel_diff_vs_fp64"] = float(np.linalg.norm(steps20[name] - steps20["fp64_products"]) /
                                                        np.linalg.norm(steps20["fp64_products"]))
    lsqr_out["mixed_speedup_vs_fp64_products"] = (lsqr_out["fp64_products"]["ms"] /
                                                  lsqr_out["mixed_factors_fp32_jacobian"]["ms"])
    s.build(c, w.k)
    J = torch.empty((w.M * w.P, w.S * w.S, 2), dtype=torch.float64, device="cuda")
    a_d, t_d = torch.tensor(al, device="cuda"), torch.tensor(th, device="cuda")
    hs.hs_jacobian_dev(s.ctx, a_d, t_d, J)
    torch.cuda.synchronize()
    # the contraction's emulated FP64 products, per-launch events
    hs.hs_prof_start(hs.HS_PROF_GEMM_EMU)
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    hs.hs_jacobian_dev(s.ctx, a_d, t_d, J)
    e1.record(stream)
    torch.cuda.synchronize()
    emu_ms, emu_flops, emu_n = hs.hs_prof_stop()
    jac_ms64 = e0.elapsed_time(e1)
    # the same Jacobian and GN step with the FP64 SIMT GEMMs (emulation off)
    hs.hs_set_fp64_emulation(False)
    J_simt = torch.empty_like(J)
    hs.hs_jacobian_dev(s.ctx, a_d, t_d, J_simt)
    torch.cuda.synchronize()
    hs.hs_prof_start(hs.HS_PROF_GEMM_FP64)
    e0.record(stream)
    hs.hs_jacobian_dev(s.ctx, a_d, t_d, J_simt)
    e1.record(stream)
    torch.cuda.synchronize()
    g_ms, g_flops, g_n = hs.hs_prof_stop()
    jac_ms_simt = e0.elapsed_time(e1)
    e0.record(stream)
    s.build(c, w.k)
    c1_simt, _ = s.gn_step(data, al, th, 1e-4, c)
    e1.record(stream)
    torch.cuda.synchronize()
    gn_ms_simt = e0.elapsed_time(e1)
    hs.hs_set_fp64_emulation(True)
    emu_vs_simt = float(torch.linalg.vector_norm(J - J_simt) / torch.linalg.vector_norm(J_simt))
    del J_simt
    s.close()
    bf16 = tf32_peak()[0] * 2.25 / 1.1
    emulated = {"kernel": "k_oz_mma (tcgen05 kind::f16, exact BF16 slices: 36 slice-pair products per FP64 product)",
                "launches": emu_n, "ms": emu_ms, "fp64_equivalent_tflops": emu_flops / (emu_ms * 1e-3) / 1e12,
                "issued_bf16_tflops": 36 * emu_flops / (emu_ms * 1e-3) / 1e12, "bf16_peak": bf16,
                "frac_issued": 36 * emu_flops / (emu_ms * 1e-3) / 1e12 / bf16,
                "peak_source": "measured bf16 burst (MEASURED_PEAKS.json)",
                "jacobian_ms_fp64_simt": jac_ms_simt, "gn_step_ms_fp64_simt": gn_ms_simt,
                "gn_step_step_rel_diff_vs_simt": float(np.linalg.norm(c1 - c1_simt) / np.linalg.norm(c1_simt - c)),
                "jacobian_rel_diff_vs_simt": emu_vs_simt}
    # the same Jacobian on a mixed-precision context (refined forward and adjoint fields, FP64
    # contraction): its time and its distance from the FP64 one
    sm = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, hs.HS_MIXED, device=local, stream=stream.cuda_stream)
    sm.build(c, w.k)
    J32 = torch.empty_like(J)
    hs.hs_jacobian_dev(sm.ctx, a_d, t_d, J32)
    torch.cuda.synchronize()
    e0.record(stream)
    hs.hs_jacobian_dev(sm.ctx, a_d, t_d, J32)
    e1.record(stream)
    torch.cuda.synchronize()
    jac_mixed = {"ms": e0.elapsed_time(e1),
                 "rel_err_vs_fp64": float(torch.linalg.vector_norm(J32 - J) / torch.linalg.vector_norm(J))}
    sm.close()
    del J, J32
    nX = 14 * w.n_leaf_side
    contract_flops = 4.0 * w.M * w.P * (nX * nX * w.S + nX * w.S * w.S)
    return {"value": float(np.median(ts)), "unit": "ms", "workload": w.name, "precision": "fp64",
            "includes": "hs_build + hs_gn_step (forward, adjoint sweep, Jacobian contraction, normal equations "
                        "Re(J^H J) + lambda I by symmetric block-row FP64 GEMMs, LU)",
            "residual_norm": float(rn), "mixed_direct": mixed_direct, "lsqr_paper_solver": lsqr_out,
            "jacobian_ms": jac_ms64, "fp64_emulation": emulated,
            "jacobian_mixed": jac_mixed,
            "jacobian_gemm_fp64": {"ms": g_ms, "launches": g_n, "tflops": g_flops / (g_ms * 1e-3) / 1e12,
                                   "contraction_algorithmic_tflop": contract_flops / 1e12}}


def run_case(name):
    """Profiler targets: 'gn_k40' = data generation and two FP64 Gauss-Newton steps of the
    k = 40 top-of-sweep workload; 'jacobian_16x16_s64' = one Jacobian at k = 20 on 16 x 16
    leaves with 64 x 64 modes and 64 x 64 data; 'lsqr_k40' = data generation and one
    LSQR Gauss-Newton step of the k = 40 workload (tolerance 1e-3, FP64 products);
    'lsqr_mixed_k40' = the same on a mixed-precision context with the tensor-core
    Jacobian, two steps."""
    import torch

    from paper_1608_06871_gb300.build import build
    build()
    import paper_1608_06871_gb300 as hs
    if name == "emulated_gemm_shapes":
        # the emulated FP64 product through hs_dgemm_emulated and the FP64 SIMT GEMM through
        # hs_zgemm on real-valued data: TFLOP/s at 2 m n k (FP64-equivalent)
        shapes = [(1, 2048, 2048, 2048), (1, 4096, 4096, 1536), (1, 262144, 64, 448), (256, 128, 64, 448)]
        g = torch.Generator(device="cuda").manual_seed(0)
        for b_, m, n, k in shapes:
            A = torch.randn((b_, m, k), dtype=torch.float64, device="cuda", generator=g)
            B = torch.randn((b_, k, n), dtype=torch.float64, device="cuda", generator=g)
            C = torch.empty((b_, m, n), dtype=torch.float64, device="cuda")
            for _ in range(2):
                hs.hs_dgemm_emulated(A, B, C)
            torch.cuda.synchronize()
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(3):
                hs.hs_dgemm_emulated(A, B, C)
            e1.record()
            torch.cuda.synchronize()
            print({"shape": [b_, m, n, k], "emulated_tflops": 2.0 * b_ * m * n * k * 3 / (e0.elapsed_time(e1) * 1e-3) / 1e12},
                  flush=True)
        return
    if name == "paper_gn_k70":
        # the paper-scale Gauss-Newton step (k = 70, 19,600 unknowns) alone, timed, as JSON
        print(json.dumps(paper_scale_gn(hs, torch, 0)), flush=True)
        return
    if name == "mixed_k20":
        # two mixed-precision build + forward calls at the k = 20 gradient workload (16 x 16 leaves,
        # 64 incidences, 128 receivers): a small target for profilers of the refinement kernels
        w = synth.WORKLOADS["grad_k20"]
        c = synth.smooth_random_coeffs(w.S, seed=2, qmax=0.3)
        s = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, hs.HS_MIXED)
        al, th = synth.directions(w.M), synth.receivers(w.P)
        for _ in range(2):
            s.build(c, w.k)
            s.solve(al, th)
        s.close()
        print("mixed_k20 done", flush=True)
        return
    if name == "lu_1792":
        # batched LU solves of complex64 systems of order 1792 (the root of the k = 40 tree)
        g = torch.Generator(device="cuda").manual_seed(0)
        A0 = torch.randn((1, 1792, 1792), dtype=torch.complex64, device="cuda", generator=g)
        B0 = torch.randn((1, 1792, 64), dtype=torch.complex64, device="cuda", generator=g)
        for _ in range(3):
            A, B = A0.clone(), B0.clone()
            hs.hs_lu_solve(A, B)
        torch.cuda.synchronize()
        print("lu_1792 done", flush=True)
        return
    if name == "jacobian_k40":
        # one FP64 Jacobian of the k = 40 top-of-sweep size (4096 modes, 160 x 160 data), after one warm-up
        w = synth.WORKLOADS["gn_k40"]
        c = np.zeros((w.S, w.S))
        c[:40, :40] = synth.project_sine(synth.ellipse_phantom(7), 40, 40)
        s = hs.Solver(w.n_leaf_side, w.S, w.S, w.R).build(c, w.k)
        a_d = torch.tensor(synth.directions(w.M), device="cuda")
        t_d = torch.tensor(synth.receivers(w.P), device="cuda")
        J = torch.empty((w.M * w.P, w.S * w.S, 2), dtype=torch.float64, device="cuda")
        for _ in range(2):
            hs.hs_jacobian_dev(s.ctx, a_d, t_d, J)
        torch.cuda.synchronize()
        print("jacobian_k40 launches", s.launch_count(), flush=True)
        s.close()
        return
    if name in ("tc_shapes", "tc_2048"):
        # FP32 products through hs_gemm32 (split-TF32 tensor-core product forced on, then the
        # SIMT FP32 GEMM): useful TFLOP/s at 8 m n k (complex), 4 m n k (real x complex),
        # 2 m n k (real); tc_2048 runs one 2048^3 complex product three times (a profiler target)
        if name == "tc_2048":
            shapes = [(2, 1, 2048, 2048, 2048)]
        else:
            shapes = [(2, 1, 2048, 2048, 2048), (2, 1, 4096, 4096, 4096), (2, 1, 1792, 1792, 1792),
                      (2, 1, 1792, 128, 3584), (2, 8, 224, 1344, 224), (2, 4, 448, 128, 896),
                      (0, 1024, 196, 196, 196), (0, 1024, 196, 56, 196), (1, 1024, 196, 128, 196),
                      (1, 1024, 56, 128, 196), (2, 1024, 56, 128, 56),
                      (2, 1, 1664, 1664, 128), (2, 1, 1024, 1024, 128), (2, 1, 512, 512, 128),
                      (2, 1, 1664, 1792, 128)]
        g = torch.Generator(device="cuda").manual_seed(0)

        def rnd(shape, cplx):
            if cplx:
                return torch.complex(torch.randn(shape, device="cuda", generator=g),
                                     torch.randn(shape, device="cuda", generator=g))
            return torch.randn(shape, device="cuda", generator=g)

        for mode, b_, m, n, k in shapes:
            A, B = rnd((b_, m, k), mode == 2), rnd((b_, k, n), mode >= 1)
            C = torch.empty((b_, m, n), dtype=torch.complex64 if mode else torch.float32, device="cuda")
            if name == "tc_2048":
                hs.hs_set_tensor_cores(2)
                for _ in range(3):
                    hs.hs_gemm32(A, B, C)
                torch.cuda.synchronize()
                hs.hs_set_tensor_cores(1)
                print("tc_2048 done", flush=True)
                return
            row = {"mode": mode, "shape": [b_, m, n, k]}
            fl = {2: 8, 1: 4, 0: 2}[mode] * b_ * m * n * k
            for label, tc in (("tc", 2), ("simt", 0)):
                hs.hs_set_tensor_cores(tc)
                for _ in range(2):
                    hs.hs_gemm32(A, B, C)
                torch.cuda.synchronize()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record()
                for _ in range(5):
                    hs.hs_gemm32(A, B, C)
                e1.record()
                torch.cuda.synchronize()
                row[label + "_tflops"] = fl * 5 / (e0.elapsed_time(e1) * 1e-3) / 1e12
            hs.hs_set_tensor_cores(1)
            print(row, flush=True)
        return
    if name in ("gn_k40", "lsqr_k40", "lsqr_mixed_k40"):
        w = synth.WORKLOADS["gn_k40"]
        ph = synth.ellipse_phantom(7)
        al, th = synth.directions(w.M), synth.receivers(w.P)
        g = hs.Solver(w.n_leaf_side, 2, 2, w.R)
        x, y = g.node_coords()
        data = synth.add_noise(g.build_nodes(ph(x, y), w.k).solve(al, th), 0.01, seed=70)
        g.close()
        c = np.zeros((w.S, w.S))
        c[:40, :40] = synth.project_sine(ph, 40, 40)
        mixed = name == "lsqr_mixed_k40"
        s = hs.Solver(w.n_leaf_side, w.S, w.S, w.R, hs.HS_MIXED if mixed else hs.HS_FP64)
        for _ in range(1 if name == "lsqr_k40" else 2):
            s.build(c, w.k)
            if name == "gn_k40":
                s.gn_step(data, al, th, 1e-4, c)
            else:
                print("lsqr iterations", s.gn_step_lsqr(data, al, th, c, tol=1e-3, max_iter=200,
                                                        products=hs.HS_MIXED if mixed else hs.HS_FP64)[2])
        torch.cuda.synchronize()
        print(name, "launches", s.launch_count())
        s.close()
    else:
        s = hs.Solver(16, 64, 64)
        s.build(synth.random_coeffs(64, 64, seed=5, scale=0.001), 20.0)
        J = s.jacobian(synth.directions(64), synth.receivers(64))
        print(name, J.shape, "launches", s.launch_count())
        s.close()


def main():
    args = parse()
    if args.case:
        run_case(args.case)
        return
    world, rank, local = dist_init()
    if args.impl == "reference":
        run_reference(args, world, rank)
    else:
        run_hs(args, world, rank, local)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
