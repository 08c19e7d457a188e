#!/usr/bin/env python
"""Benchmark of the GMG-preconditioned FGMRES slab solve on one GB300 (or N replicas).

Step = one flexible-GMRES solve (V(2,2) additive-Vanka V-cycle per iteration) of the dG(k)
Q2/P1disc slab Newton system to 1e-8 relative residual, from x = 0, with the hierarchy assembled
and factored once beforehand (assembly and factorisation times are reported under "setup").
Default workload: the 3D channel with a square-prism obstacle, 3 levels (fine 64x16x16 minus the
obstacle), dG(1), 962,208 DoFs, cell inverses of 170x170.

The headline `value` is seconds per solve of the fastest mixed-precision run whose V-cycle keeps
every residual product in FP64: cell inverses stored and applied in FP32 or BF16 (FP32
accumulation), FP64 FGMRES, Arnoldi, residual products and coarse solve. The plain FP64 path is
timed in the same run ("fp64_s"); every precision reports its error against the FP64 solution.
A run with FP32 V-cycle defects ("bf16+f32d") is reported as an extra row only.

Prints ONE JSON line (rank 0). `--impl reference` times the CPU oracle (the plain FP64 reference
implementation written from the paper) on a bounded sample of the same workload instead.
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

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

DEFAULT_WORKLOAD = "c3_3d_k1"
# conforming mixed-precision arms (FP64 residual products): the headline is the fastest of these
CONFORMING_MIXED = ("f32", "bf16")


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["gpu", "reference"], default="gpu")
    ap.add_argument("--workload", default=DEFAULT_WORKLOAD)
    ap.add_argument("--rtol", type=float, default=1e-8)
    ap.add_argument("--precisions", default="f64,f32,bf16,bf16+f32d",
                    help="cell-inverse storage per run; INV+f32d also takes the V-cycle defects in FP32")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-other-rows", action="store_true", help="skip the other-workload rows (c2, c5)")
    ap.add_argument("--multi-restart", type=int, default=20)
    ap.add_argument("--robustness", action="store_true",
                    help="viscosity / damping study: Newton and FGMRES counts for nu x omega_d (V(4,4), tau 0.005)")
    ap.add_argument("--march", type=int, default=0,
                    help="time-march this many slabs (damped Newton per slab) and report the wake functional")
    ap.add_argument("--mesh-study", action="store_true",
                    help="FGMRES iterations of V(1,1) and V(4,4) as one coarse grid is refined (2D and 3D dG(1))")
    ap.add_argument("--newton", action="store_true",
                    help="time the damped Newton solve of the nonlinear slab problem instead of one linear solve")
    ap.add_argument("--kernel-driver", choices=["product_sweep", "multi_sweep", "fused_sweep", "coarse"], default=None,
                    help="small fixed launch sequence for a profiler: the finest-level FP64 product and single-RHS "
                         "sweep, the 32-column or fused 16+16 sweep, or the coarse solve, --steps times each")
    ap.add_argument("--levels", type=int, default=0, help="override the workload's number of levels")
    ap.add_argument("--oracle-child", default=None, help=argparse.SUPPRESS)
    return ap.parse_args()


def workload(name):
    import synth

    return synth.WORKLOADS[name]


def describe(wl, sizes):
    fine = sizes[-1]
    return {"workload": f"{wl.name}: {wl.dim}D channel {'x'.join(map(str, wl.fine_cells))} fine cells "
                        f"({'obstacle' if wl.obstacle_lo != wl.obstacle_hi else 'no obstacle'}), "
                        f"{wl.n_levels} levels, Q2/P1disc x dG({wl.k})",
            "dofs": fine["n_dofs"], "cells": fine["n_cells"], "n_local": fine["n_local"],
            "levels": wl.n_levels, "rtol": None, "smoother": f"additive Vanka V({wl.nu1},{wl.nu2}) omega={wl.omega}",
            "krylov": f"FGMRES({wl.restart})", "nu": wl.nu, "tau": wl.tau}


# ---------------------------------------------------------------------------------------------
# CPU oracle leg (run in spawned child processes so that it never shares the CUDA context)
# ---------------------------------------------------------------------------------------------
# The oracle's set-up of the full 3D workload takes minutes (numpy assembly, Python-loop transfer
# matrices, a sparse LU of the coarse level), so the CPU baseline runs on a bounded sample: the same
# channel, element pair, time degree, obstacle rule and seeded data with one refinement level fewer
# (config 3 on 2 levels: 127,920 DoFs), scaled to the full workload by the ratio of DoFs (one FGMRES
# iteration costs O(DoFs); the iteration count does not depend on the mesh, Tables 5.1 / 5.5).
SAMPLE_LEVELS_DROP = 1
REFERENCE_MAX_STEPS = 8


def oracle_child(spec_path):
    spec = json.load(open(spec_path))
    if spec.get("cpus") and hasattr(os, "sched_setaffinity"):
        os.sched_setaffinity(0, set(spec["cpus"]))
    import dataclasses

    import numpy as np

    import synth
    from oracle import solvers

    wl = synth.WORKLOADS[spec["workload"]]
    if spec.get("n_levels"):
        wl = dataclasses.replace(wl, n_levels=spec["n_levels"])
    t0 = time.perf_counter()
    H = solvers.Hierarchy(wl, synth.linearisation_point(wl))
    setup = time.perf_counter() - t0
    lev = H.fine
    rng = np.random.default_rng(7)
    r, d = rng.standard_normal(lev.N), rng.standard_normal(lev.N)
    sweep_s = []
    for _ in range(spec.get("sweeps", 0)):
        t0 = time.perf_counter()
        solvers.vanka_step(lev, H.J[-1], H.inv[-1], d, r, wl.omega)
        sweep_s.append(time.perf_counter() - t0)
    b = lev.dofs_from_lattice(synth.random_rhs(wl))
    times, iters = [], []
    x, info = None, {"converged": False}
    for _ in range(spec["solves"]):
        t0 = time.perf_counter()
        x, info = H.solve(b, rtol=spec["rtol"], maxit=spec["maxit"])
        times.append(time.perf_counter() - t0)
        iters.append(info["iters"])
    if spec.get("x_out") and x is not None:
        np.save(spec["x_out"], x)
    sizes = {"n_dofs": int(lev.N), "n_cells": int(lev.C), "n_local": int(lev.n), "n_levels": wl.n_levels}
    json.dump({"setup_s": setup, "solve_s": times, "iters": iters, "converged": bool(info["converged"]),
               "sweep_s": sweep_s, "sizes": sizes}, open(spec["out"], "w"))


def start_oracle(wl_name, rtol, solves, sweeps=0, n_levels=None, threads=1, maxit=1000, x_out=None, cpus=None):
    """Spawn the oracle child; returns a handle for finish_oracle (the child runs while the caller
    does other work)."""
    td = tempfile.mkdtemp(prefix="stm_oracle_")
    spec = {"workload": wl_name, "rtol": rtol, "solves": solves, "sweeps": sweeps, "maxit": maxit,
            "n_levels": n_levels, "out": os.path.join(td, "o.json"), "x_out": x_out, "cpus": cpus}
    sp = os.path.join(td, "spec.json")
    json.dump(spec, open(sp, "w"))
    env = dict(os.environ)
    for v in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        env[v] = str(threads)
    env["CUDA_VISIBLE_DEVICES"] = ""
    proc = subprocess.Popen([sys.executable, os.path.abspath(__file__), "--oracle-child", sp], env=env,
                            stdout=subprocess.DEVNULL, stderr=subprocess.PIPE, text=True)
    return {"proc": proc, "spec": spec, "dir": td, "threads": threads}


def finish_oracle(handle):
    import shutil

    err = handle["proc"].communicate()[1]
    try:
        if handle["proc"].returncode != 0:
            raise RuntimeError("oracle child failed:\n" + (err or "")[-3000:])
        out = json.load(open(handle["spec"]["out"]))
        out["threads"] = handle["threads"]
        return out
    finally:
        shutil.rmtree(handle["dir"], ignore_errors=True)


def run_oracle(wl_name, rtol, solves, maxit=1000, threads=1, n_levels=None, sweeps=0):
    return finish_oracle(start_oracle(wl_name, rtol, solves, sweeps=sweeps, n_levels=n_levels, threads=threads,
                                      maxit=maxit))


def cpu_model():
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.strip().startswith("Model name:"):
                return line.split(":", 1)[1].strip()
    except (OSError, subprocess.SubprocessError):
        pass
    import platform

    return platform.processor() or platform.machine()


def sample_levels(wl):
    return max(2, wl.n_levels - SAMPLE_LEVELS_DROP)


def cpu_baseline_entry(o1, on, full_dofs, full_cells, gpu_iters, wl):
    """cpu_baseline of the bench line from the 1-thread and all-thread oracle samples."""
    import numpy as np

    scale = full_dofs / o1["sizes"]["n_dofs"]
    cscale = full_cells / o1["sizes"]["n_cells"]

    def leg(o):
        return {"threads": o["threads"], "solve_s_sample_median": float(np.median(o["solve_s"])),
                "solve_s_scaled": float(np.median(o["solve_s"])) * scale, "iters_sample": o["iters"][-1],
                "sweep_s_sample_median": float(np.median(o["sweep_s"])) if o["sweep_s"] else None,
                "sweep_s_scaled": float(np.median(o["sweep_s"])) * cscale if o["sweep_s"] else None,
                "setup_s_sample_untimed": o["setup_s"]}

    one, alln = leg(o1), leg(on)
    return {"value": one["solve_s_scaled"], "unit": "s", "cores": 1, "kind": "oracle",
            "sample": (f"the oracle's full FP64 FGMRES solve (rtol {wl.rtol:g}) of the same 3D dG(1) channel with one "
                       f"refinement level fewer ({o1['sizes']['n_levels']} levels, {o1['sizes']['n_dofs']:,} DoFs, "
                       f"{o1['iters'][-1]} iterations; the GPU needs {gpu_iters} on the full workload), median of "
                       f"{len(o1['solve_s'])}, scaled by the DoF ratio {scale:.3f}; the Vanka sweep (the oracle's "
                       f"vanka_step: residual, local solves, weighted combine) on that sample's finest level "
                       f"({o1['sizes']['n_cells']:,} cells, n = {o1['sizes']['n_local']}), median of "
                       f"{len(o1['sweep_s'])}, scaled by the cell ratio {cscale:.3f}"),
            "cpu_model": cpu_model(), "nproc": os.cpu_count(), "cores_all_threads_leg": on["threads"],
            "one_thread": one, "all_threads": alln,
            "note": "numpy/scipy as written: the sparse products, einsum local solves and the SuperLU coarse "
                    "solve run on one thread whatever the BLAS thread count"}


# ---------------------------------------------------------------------------------------------
# clocks sampled during the timed region
# ---------------------------------------------------------------------------------------------
class ClockSampler:
    QUERY = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
             "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
             "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.proc = None
        self.gpu = gpu_index
        self.path = tempfile.mktemp(suffix=".csv")

    def start(self):
        try:
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.QUERY}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=self.fh, stderr=subprocess.DEVNULL)
        except (OSError, FileNotFoundError):
            self.proc = None

    def stop(self):
        if self.proc is None:
            return None
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.fh.close()
        rows = []
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                rows.append(dict(sm=float(parts[1]), smax=float(parts[2]), hw=parts[5], hwt=parts[6], swt=parts[7],
                                 pcap=parts[8]))
            except ValueError:
                continue
        os.remove(self.path)
        if not rows:
            return None
        reasons = set()
        for r in rows:
            for key, name in (("hw", "hw_slowdown"), ("hwt", "hw_thermal_slowdown"), ("swt", "sw_thermal_slowdown"),
                              ("pcap", "sw_power_cap")):
                if r[key].lower() == "active":
                    reasons.add(name)
        return {"sm_mhz": statistics.median(r["sm"] for r in rows), "sm_max_mhz": max(r["smax"] for r in rows),
                "reasons": sorted(reasons), "samples": len(rows)}


def recorded_traffic(workload_name, kernel, prec=None):
    """DRAM bytes per launch of a finest-level kernel from a committed ncu capture, valid only
    while the kernel's source file is unchanged since the capture (sha256 of the file)."""
    import hashlib

    try:
        rec = json.load(open(os.path.join(ROOT, "profiles", "roofline_traffic.json")))
    except (OSError, ValueError):
        return None
    for e in rec.get("captures", []):
        if e.get("workload") != workload_name or e.get("kernel") != kernel:
            continue
        if prec is not None and e.get("precision") not in (prec, "any"):
            continue
        try:
            sha = hashlib.sha256(open(os.path.join(ROOT, e["source"]), "rb").read()).hexdigest()
        except (OSError, KeyError):
            continue
        if sha == e.get("source_sha256"):
            return {"per_launch_bytes": e["dram_bytes_read"] + e["dram_bytes_write"], "source": e["profile"]}
    return None


def spmv_roofline(r, wl, sizes, fp64_peak, workload_name, hbm=None, peak_source=None):
    """Dominant kernel of the solve: the product with the finest J in FP64 accuracy.

    Over FP64 values (small 2D levels) the FP64 pipe is the bound: achieved = 2 * nnz FLOP per launch (one
    FMA per stored value) / average event time per launch; peak = FP64 FMA throughput measured in the same
    run (stm_measure_fp64_peak). With hbm given, the level keeps two-limb integers and its bytes are the
    bound: achieved = algorithmic bytes per launch / the same time, peak = the measured copy bandwidth."""
    f = r["finest"]["jacobian_spmv"]
    if f["ms"] <= 0 or f["launches"] == 0:
        return None
    nnz = sizes[-1]["nnz"]
    us = 1e3 * f["ms"] / f["launches"]
    achieved = 2.0 * nnz / (us * 1e-6) / 1e12
    if hbm:
        traffic = recorded_traffic(workload_name, "k_spmv_limbs")
        gbs = f["bytes"] / (f["ms"] * 1e-3) / 1e9
        return {"kernel": "k_spmv_limbs (J_g x, finest level, two-limb integers with the exponents of x)",
                "bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
                "traffic": traffic["per_launch_bytes"] if traffic else None,
                "traffic_source": traffic["source"] if traffic else "no capture of the current kernel source",
                "peak_source": peak_source, "avg_launch_us": us, "fp64_tflops_equivalent": achieved,
                "fp64_pipe_tflops": fp64_peak, "algorithmic_bytes_per_launch": f["bytes"] / f["launches"]}
    traffic = recorded_traffic(workload_name, "k_spmv_nb_dyn")
    return {"kernel": "k_spmv_nb_dyn (J_g x, finest level, FP64)", "bound": "alu", "achieved": achieved,
            "peak": fp64_peak, "unit": "TFLOP/s", "frac": achieved / fp64_peak if fp64_peak else None,
            "traffic": traffic["per_launch_bytes"] if traffic else None,
            "traffic_source": traffic["source"] if traffic else "no capture of the current kernel source",
            "peak_source": "FP64 FMA rate measured in this run (stm_measure_fp64_peak)",
            "flops_per_launch": 2.0 * nnz, "avg_launch_us": us,
            "algorithmic_bytes_per_launch": f["bytes"] / f["launches"],
            "hbm_gbs_algorithmic": f["bytes"] / (f["ms"] * 1e-3) / 1e9}


def limb_hbm(wl, hbm=None):
    """The copy bandwidth where the workload's finest level keeps two-limb integers (3D), else None."""
    if wl.dim != 3:
        return None
    if hbm is None:
        pk = peaks()
        hbm = pk["hbm_gbs"] if pk else 6800.0
    return hbm


def defect_roofline(r, sizes, hbm, peak_source, workload_name):
    """The V-cycle's defect r - J_g d over the FP32 copies of J_g, finest level (HBM bound).

    achieved = (4 nnz + 20 N) algorithmic bytes per launch (FP32 values and d, FP64 r and t) / average
    event time per launch of the product kernel; peak = the measured copy bandwidth. The rounding of
    d to FP32 before it (12 N bytes, a launch of its own) is timed as class round_f32."""
    f = r["finest"]["defect_f32"]
    if f["ms"] <= 0 or f["launches"] == 0:
        return None
    us = 1e3 * f["ms"] / f["launches"]
    by = f["bytes"] / f["launches"]
    achieved = by / (us * 1e-6) / 1e9
    traffic = recorded_traffic(workload_name, "k_spmv_nodeblock_f32")
    return {"kernel": "k_spmv_nodeblock<float> (r - J_g d over FP32 values, finest level)", "bound": "hbm",
            "achieved": achieved, "peak": hbm, "unit": "GB/s", "frac": achieved / hbm,
            "traffic": traffic["per_launch_bytes"] if traffic else None,
            "traffic_source": traffic["source"] if traffic else "no capture of the current kernel source",
            "peak_source": peak_source, "bytes_per_launch": by, "avg_launch_us": us}


def spmm_roofline(f, nnz, kern, workload_name):
    """The multi-RHS SpMM Y = J_g X (32 columns) in FP64 accuracy, finest level, against the copy bandwidth.

    On the workload it is quoted for the product runs on the tensor cores over base-256 digits and is bound by
    chains of dependent instructions (forming digits, joining sums). achieved = algorithmic bytes (J once, X and Y once) per launch / average
    event time per launch; peak = measured copy bandwidth; fp64_tflops_equivalent = 2 * nnz * 32 FLOP over the
    same time; share = the finest-level SpMM event time over the event time of all classes in the profiled solve."""
    if f["ms"] <= 0 or f["launches"] == 0:
        return None
    us = 1e3 * f["ms"] / f["launches"]
    pk = peaks()
    hbm = pk["hbm_gbs"] if pk else 6800.0
    gbs = f["bytes"] / (f["ms"] * 1e-3) / 1e9
    total = sum(v["ms"] for v in kern.values())
    traffic = recorded_traffic(workload_name, "k_spmm_digits")
    return {"kernel": "k_spmm_digits (Y = J_g X, 32 columns, finest level)", "bound": "latency",
            "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
            "traffic": traffic["per_launch_bytes"] if traffic else None,
            "traffic_source": traffic["source"] if traffic else "no capture of the current kernel source",
            "peak_source": "MEASURED_PEAKS.json hbm_gbs" if pk else "fallback 6.8 TB/s",
            "fp64_tflops_equivalent": 2.0 * nnz * 32 / (us * 1e-6) / 1e12,
            "algorithmic_bytes_per_launch": f["bytes"] / f["launches"], "avg_launch_us": us,
            "launches_per_solve": f["launches"], "share_of_profiled_solve": f["ms"] / total if total > 0 else None}


def max_over_ranks(value, dist, device):
    """Replicas (one independent slab solve per GPU): the job's time per step is the slowest rank's."""
    import torch

    t = torch.tensor([float(value)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def mode_precision(args):
    """Precision of the single-precision study modes (Newton, marching, mesh and robustness studies):
    the last requested one whose V-cycle defects stay FP64, else the last one."""
    toks = args.precisions.split(",")
    keep = [t for t in toks if "+f32d" not in t]
    return keep[-1] if keep else toks[-1]


def split_precision(tok):
    """'bf16+f32d' -> ('bf16', 'f32'): cell-inverse storage and V-cycle defect precision."""
    inv, sep, d = tok.partition("+")
    if inv not in ("f64", "f32", "bf16") or (sep and d != "f32d"):
        raise ValueError(f"precision {tok!r}: expected f64|f32|bf16, optionally +f32d")
    return inv, ("f32" if d else "f64")


def hier_params(wl, tok, smoother="additive"):
    from paper_2107_10561_gb300 import make_params

    inv, dp = split_precision(tok)
    return make_params(wl.dim, wl.k, wl.n_levels, wl.coarse_cells, wl.length, wl.obstacle_lo, wl.obstacle_hi,
                       wl.tau, wl.nu, wl.gamma1, wl.gamma2, inv, smoother, wl.omega, wl.nu1, wl.nu2,
                       defect_precision=dp)


def dtype_label(tok):
    inv, dp = split_precision(tok)
    if inv == "f64" and dp == "f64":
        return "f64"
    parts = [f"{inv} cell inverses (f32 accumulate)"] if inv != "f64" else []
    if dp == "f32":
        parts.append("f32 V-cycle defects")
    return "f64 Krylov/Arnoldi SpMV/coarse + " + " + ".join(parts)


def peaks():
    try:
        return json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except OSError:
        return None


# ---------------------------------------------------------------------------------------------
# GPU leg
# ---------------------------------------------------------------------------------------------
def lattice_vec(h, arr):
    import numpy as np
    import torch

    idx = h.dof_lattice_index()
    return torch.from_numpy(np.ascontiguousarray(arr.reshape(-1)[idx])).cuda()


def time_precisions(wl, precs, state, rhs_lat, steps, warmup, rtol, dist=None, profile=True):
    """Per precision token: build, assemble, factor, W warm-up solves, then K timed solves from x = 0
    (CUDA events on the launching stream, V-cycles replayed as CUDA graphs), then the same K solves
    with per-kernel event timing (direct launches). Returns (results, hierarchies)."""
    import torch

    from paper_2107_10561_gb300 import Hierarchy

    results, hs = {}, {}
    for prec in precs:
        h = Hierarchy(hier_params(wl, prec, "additive"))
        X = lattice_vec(h, state)
        b = lattice_vec(h, rhs_lat)
        e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
        torch.cuda.synchronize()
        e0.record()
        h.assemble_jacobian(X)
        e1.record()
        h.factor_cells()
        e2.record()
        torch.cuda.synchronize()
        setup = {"assemble_ms": e0.elapsed_time(e1), "factor_ms": e1.elapsed_time(e2)}
        x = torch.zeros_like(b)
        info = None
        for _ in range(warmup):
            x.zero_()
            info = h.gmres_solve(b, x, rtol=rtol, restart=wl.restart)
        hs[prec] = (h, b, x)
        results[prec] = {"setup": setup}
    stream = torch.cuda.current_stream()
    for prec, (h, b, x) in hs.items():
        launches0 = Hierarchy.kernel_launches()
        if dist:
            dist.barrier()
        torch.cuda.synchronize()
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.nvtx.range_push(f"timed_solves_{prec.replace('+', '_')}")  # lets a profiler select these launches
        ev0.record(stream)
        for _ in range(steps):
            x.zero_()
            info = h.gmres_solve(b, x, rtol=rtol, restart=wl.restart)
        ev1.record(stream)
        torch.cuda.nvtx.range_pop()
        torch.cuda.synchronize()
        ms = ev0.elapsed_time(ev1) / steps
        if dist:
            ms = max_over_ranks(ms, dist, "cuda")
        r = results[prec]
        r["ms_per_solve"] = ms
        r["launches_per_step"] = (Hierarchy.kernel_launches() - launches0) / steps
        r["iters_timed"] = info["iters"]
        r["rel_res_true_timed"] = info["rel_res_true"]
        r["graphs_timed"] = info.get("graphs")
        if not profile:
            continue
        # profiled pass over the same steps: CUDA events around every launch of the library, recorded
        # on the launching stream (direct launches, no graphs), for the per-kernel split and roofline
        h.profile_enable(True)
        torch.cuda.synchronize()
        pv0, pv1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        pv0.record(stream)
        for _ in range(steps):
            x.zero_()
            h.gmres_solve(b, x, rtol=rtol, restart=wl.restart)
        pv1.record(stream)
        torch.cuda.synchronize()
        r["ms_per_solve_profiled"] = pv0.elapsed_time(pv1) / steps
        r["kernels"] = {k: h.profile_read(k) for k in ("vanka_local", "jacobian_spmv", "defect_f32", "round_f32",
                                                       "vanka_combine", "transfer", "coarse", "krylov")}
        r["finest"] = {k: h.profile_read(k, wl.n_levels - 1) for k in ("vanka_local", "jacobian_spmv", "defect_f32")}
        r["per_level"] = {k: [h.profile_read(k, g) for g in range(wl.n_levels)]
                          for k in ("vanka_local", "jacobian_spmv", "defect_f32", "vanka_combine", "transfer")}
        h.profile_enable(False)
    return results, hs


def solution_errors(hs, ref="f64"):
    """Error of every precision's solution against the FP64 solution of the same run (same b)."""
    if ref not in hs:
        return {}
    xr = hs[ref][2].double()
    nr_max, nr_2 = float(xr.abs().max()), float(xr.norm())
    out = {}
    for p, (_, _, x) in hs.items():
        dx = x.double() - xr
        out[p] = {"max_rel": float(dx.abs().max()) / nr_max, "l2_rel": float(dx.norm()) / nr_2}
    return out


def by_precision_rows(results, errs, steps):
    def gbs(e):
        return e["bytes"] / (e["ms"] * 1e-3) / 1e9 if e["ms"] > 0 else None

    def us(e):
        return 1e3 * e["ms"] / e["launches"] if e["launches"] else None

    out = {}
    for p, v in results.items():
        inv, dp = split_precision(p)
        row = {"s_per_solve": v["ms_per_solve"] / 1e3, "iters": v["iters_timed"],
               "rel_res_true": v["rel_res_true_timed"], "vcycle_graphs": v.get("graphs_timed"),
               "setup_ms": v["setup"],
               "fp64_residual_products": dp == "f64",
               "err_vs_fp64_solution": errs.get(p)}
        if dp != "f64":
            row["note"] = ("extra row: FP32 V-cycle defects, outside the rule that the residual products "
                           "stay FP64; not a headline candidate")
        if "kernels" in v:
            k, f = v["kernels"], v["finest"]
            row.update({"vanka_sweep_gbs": gbs(k["vanka_local"]), "spmv_gbs": gbs(k["jacobian_spmv"]),
                        "finest_vanka_gbs": gbs(f["vanka_local"]), "finest_spmv_gbs": gbs(f["jacobian_spmv"]),
                        "finest_vanka_us": us(f["vanka_local"]), "finest_spmv_us": us(f["jacobian_spmv"]),
                        "finest_defect_f32_us": us(f["defect_f32"]), "finest_defect_f32_gbs": gbs(f["defect_f32"]),
                        "kernel_ms_per_solve": {kk: kv["ms"] / steps for kk, kv in k.items()},
                        "us_per_launch_by_level": {kk: [round(1e3 * e["ms"] / e["launches"], 2) if e["launches"] else None
                                                        for e in lv] for kk, lv in v["per_level"].items()},
                        "s_per_solve_profiled_pass": v["ms_per_solve_profiled"] / 1e3})
        out[p] = row
    return out


def pick_head(results):
    mixed = [p for p in CONFORMING_MIXED if p in results]
    return min(mixed, key=lambda p: results[p]["ms_per_solve"]) if mixed else next(iter(results))


def gpu_leg(args, rank, world, local_rank):
    import torch

    import synth
    from paper_2107_10561_gb300 import Hierarchy
    from paper_2107_10561_gb300 import build as _build

    torch.cuda.set_device(local_rank)
    dist = None
    if world > 1:
        import torch.distributed as dist

        dist.init_process_group("nccl")
    _build.build()
    wl = workload(args.workload)
    state = synth.linearisation_point(wl)
    rhs_lat = synth.random_rhs(wl, seed_offset=rank)
    precs = args.precisions.split(",")
    sampler = ClockSampler(local_rank)
    sampler.start()
    time.sleep(0.3)
    results, hs = time_precisions(wl, precs, state, rhs_lat, args.steps, args.warmup, args.rtol, dist)
    clocks = sampler.stop()
    sizes = [hs[precs[0]][0].sizes(g) for g in range(wl.n_levels)]
    fp64_peak = Hierarchy.measure_fp64_peak()
    errs = solution_errors(hs)
    head = pick_head(results)
    # end-to-end through the host-buffer entry point (H2D of b, D2H of x inside the timed region)
    h, b, x = hs[head]
    bh = b.cpu().pin_memory()
    xh = torch.zeros_like(bh).pin_memory()
    h.gmres_solve_host(bh, xh, rtol=args.rtol, restart=wl.restart)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        h.gmres_solve_host(bh, xh, rtol=args.rtol, restart=wl.restart)
    torch.cuda.synchronize()
    e2e_s = (time.perf_counter() - t0) / args.steps
    rows = other_rows(args, wl, hs, head, state, rhs_lat) if rank == 0 else {}
    for hh, _, _ in hs.values():
        hh.close()
    hs.clear()
    torch.cuda.empty_cache()
    return wl, sizes, results, errs, head, clocks, e2e_s, dist, fp64_peak, rows


def other_rows(args, wl, hs, head, state, rhs_lat):
    """Timings of the rows that the headline solve does not isolate, on the same workload and the
    head precision: one V-cycle (Algorithm 1, direct launches), the adjoint solve J^T lambda = b
    (transposed Vanka, P/P^T, coarse inverse^T), and the solve with the coloured multiplicative and
    the literal overwrite smoother (Sec. 4.2)."""
    import torch

    from paper_2107_10561_gb300 import Hierarchy

    out = {}
    h, b, x = hs[head]
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    d = torch.zeros_like(b)
    h.vcycle(b, d)
    torch.cuda.synchronize()
    ev0.record()
    for _ in range(10):
        h.vcycle(b, d)
    ev1.record()
    torch.cuda.synchronize()
    out["vcycle_ms"] = ev0.elapsed_time(ev1) / 10
    x.zero_()
    h.gmres_solve(b, x, rtol=args.rtol, restart=wl.restart, transpose=True)  # warm-up (J^T values)
    torch.cuda.synchronize()
    ev0.record()
    for _ in range(args.steps):
        x.zero_()
        info = h.gmres_solve(b, x, rtol=args.rtol, restart=wl.restart, transpose=True)
    ev1.record()
    torch.cuda.synchronize()
    out["adjoint_solve"] = {"ms": ev0.elapsed_time(ev1) / args.steps, "iters": info["iters"],
                            "rel_res_true": info["rel_res_true"], "precision": head}
    for smoother in ("coloured", "overwrite"):
        hv = Hierarchy(hier_params(wl, head, smoother))
        X = lattice_vec(hv, state)
        bv = lattice_vec(hv, rhs_lat)
        hv.assemble_jacobian(X)
        hv.factor_cells()
        xv = torch.zeros_like(bv)
        hv.gmres_solve(bv, xv, rtol=args.rtol, restart=wl.restart, raise_on_fail=False)
        torch.cuda.synchronize()
        ev0.record()
        for _ in range(args.steps):
            xv.zero_()
            info = hv.gmres_solve(bv, xv, rtol=args.rtol, restart=wl.restart, raise_on_fail=False)
        ev1.record()
        torch.cuda.synchronize()
        out[f"{smoother}_solve"] = {"ms": ev0.elapsed_time(ev1) / args.steps, "iters": info["iters"],
                                    "converged": info["status"] == "STM_OK", "precision": head}
        hv.close()
    return out


def workload_row(args, name, precs, steps, warmup):
    """Another single-right-hand-side workload at the same settings: seconds per solve per precision,
    errors against its FP64 solution, and the finest-level FP64 product against the FP64 rate."""
    import torch

    import synth
    from paper_2107_10561_gb300 import Hierarchy

    wl = workload(name)
    results, hs = time_precisions(wl, precs, synth.linearisation_point(wl), synth.random_rhs(wl), steps, warmup,
                                  args.rtol)
    sizes = [hs[precs[0]][0].sizes(g) for g in range(wl.n_levels)]
    errs = solution_errors(hs)
    for hh, _, _ in hs.values():
        hh.close()
    torch.cuda.empty_cache()
    head = pick_head(results)
    fp64_peak = Hierarchy.measure_fp64_peak()
    row = {"workload": describe(wl, sizes)["workload"], "dofs": sizes[-1]["n_dofs"], "rtol": args.rtol,
           "head": head, "s_per_solve": results[head]["ms_per_solve"] / 1e3,
           "fp64_s": results["f64"]["ms_per_solve"] / 1e3 if "f64" in results else None,
           "by_precision": by_precision_rows(results, errs, steps),
           "roofline_spmv_f64": {p: spmv_roofline(results[p], wl, sizes, fp64_peak, name, limb_hbm(wl), "hbm_gbs")
                                 for p in results
                                 if split_precision(p)[1] == "f64"}}
    return row


def oracle_sample_check(args, wl, precs, x_oracle):
    """Every precision's GPU solution against the oracle's FP64 solution on the bounded oracle sample
    (the same workload with one refinement level fewer): max |x - x_oracle| / max |x_oracle|."""
    import dataclasses

    import numpy as np
    import torch

    import synth
    from paper_2107_10561_gb300 import Hierarchy

    ws = dataclasses.replace(wl, n_levels=sample_levels(wl))
    state, rhs = synth.linearisation_point(ws), synth.random_rhs(ws)
    out = {}
    for prec in precs:
        h = Hierarchy(hier_params(ws, prec, "additive"))
        h.assemble_jacobian(lattice_vec(h, state))
        h.factor_cells()
        b = lattice_vec(h, rhs)
        x = torch.zeros_like(b)
        info = h.gmres_solve(b, x, rtol=args.rtol, restart=ws.restart)
        xg = x.cpu().numpy()
        out[prec] = {"max_rel": float(np.abs(xg - x_oracle).max() / np.abs(x_oracle).max()),
                     "l2_rel": float(np.linalg.norm(xg - x_oracle) / np.linalg.norm(x_oracle)),
                     "iters": info["iters"]}
        h.close()
    return out


def unique_sweep_bytes(size, prec):
    """HBM bytes a 32-column local-product launch must move at least: inverses as stored (n x ld per
    cell), index map, the residual block once (packed BF16 hi/lo pairs, 4 bytes per value, for BF16
    inverses on the tensor cores; FP64 otherwise), the results (FP32; FP64 with FP64 inverses)."""
    s = {"f64": 8, "f32": 4, "bf16": 2}[prec]
    n, C, N = size["n_local"], size["n_cells"], size["n_dofs"]
    v = 16 // s
    ld = -(-n // v) * v
    t_bytes = 4 if prec == "bf16" else 8
    return C * n * ld * s + 4 * C * n + 32 * t_bytes * N + C * n * 32 * (8 if prec == "f64" else 4)


def multi_row(args, name, steps, warmup, prec="bf16"):
    """Multi-RHS workload: 32 right-hand sides b(U_j, nu) + c(w, w) sharing one hierarchy; seconds per
    32-column solve and the finest-level multi-RHS Vanka sweep against HBM."""
    import numpy as np
    import torch

    import synth
    from paper_2107_10561_gb300 import Hierarchy

    wl = workload(name)
    nrhs = wl.extra["nrhs"]
    t0 = time.perf_counter()
    h = Hierarchy(hier_params(wl, prec, "additive"))
    build_s = time.perf_counter() - t0
    X = lattice_vec(h, synth.linearisation_point(wl))
    e0, e1, e2 = (torch.cuda.Event(enable_timing=True) for _ in range(3))
    torch.cuda.synchronize()
    e0.record()
    h.assemble_jacobian(X)
    e1.record()
    h.factor_cells()
    e2.record()
    torch.cuda.synchronize()
    n = h.n_dofs()
    B = torch.empty((nrhs, n), dtype=torch.float64, device="cuda")
    for c, U in enumerate(synth.inflow_sweep(nrhs)):
        h.assemble_rhs(float(U), wl.nu, B[c], which=0)
    Xs = torch.zeros_like(B)
    infos = None
    for _ in range(warmup):
        Xs.zero_()
        infos = h.gmres_solve_multi(B, Xs, rtol=args.rtol, restart=args.multi_restart)
    launches0 = Hierarchy.kernel_launches()
    torch.cuda.synchronize()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record()
    for _ in range(steps):
        Xs.zero_()
        infos = h.gmres_solve_multi(B, Xs, rtol=args.rtol, restart=args.multi_restart)
    ev1.record()
    torch.cuda.synchronize()
    ms = ev0.elapsed_time(ev1) / steps
    launches = Hierarchy.kernel_launches() - launches0
    h.profile_enable(True)
    Xs.zero_()
    h.gmres_solve_multi(B, Xs, rtol=args.rtol, restart=args.multi_restart)
    kern = {k: h.profile_read(k) for k in ("vanka_local", "jacobian_spmv", "vanka_combine", "transfer", "coarse",
                                           "krylov")}
    fin = h.profile_read("vanka_local", wl.n_levels - 1)
    fin_spmm = h.profile_read("jacobian_spmv", wl.n_levels - 1)
    h.profile_enable(False)
    sizes = [h.sizes(g) for g in range(wl.n_levels)]
    # one smoothing step on the finest level: 32 forward columns, and 16 forward + 16 adjoint columns
    # from one pass over the inverses (stm_vanka_sweep_fused); local products timed by event pairs
    gf = wl.n_levels - 1
    nf = sizes[-1]["n_dofs"]
    R = torch.randn(32, nf, dtype=torch.float64, device="cuda")
    D = torch.zeros_like(R)
    sweeps = {}
    for kind in ("forward_32", "fused_16_16"):
        def one():
            if kind == "forward_32":
                h.vanka_sweep_multi(gf, R, D)
            else:
                h.vanka_sweep_fused(gf, R[:16], D[:16], R[16:], D[16:])
        one()
        h.profile_enable(True)
        for _ in range(3):
            one()
        loc = h.profile_read("vanka_local", gf)
        h.profile_enable(False)
        sweeps[kind] = {"local_us": 1e3 * loc["ms"] / max(loc["launches"], 1),
                        "local_gbs_unique": unique_sweep_bytes(sizes[-1], "bf16") / (loc["ms"] / max(loc["launches"], 1) * 1e-3) / 1e9}
    h.close()
    torch.cuda.empty_cache()
    pk = peaks()
    hbm = pk["hbm_gbs"] if pk else 6800.0
    ub = unique_sweep_bytes(sizes[-1], prec)
    us_fin = 1e3 * fin["ms"] / max(fin["launches"], 1)
    ach = ub / (us_fin * 1e-6) / 1e9 if fin["ms"] > 0 else None
    spmm = spmm_roofline(fin_spmm, sizes[-1]["nnz"], kern, name)
    vanka = {"kernel": f"k_vanka_mrhs_tc5 (multi-RHS Vanka local products, {prec} inverses on tcgen05), "
                       f"finest level, 32 columns", "bound": "hbm",
             "achieved": ach, "peak": hbm, "unit": "GB/s", "frac": ach / hbm if ach else None,
             "avg_launch_us": us_fin, "bytes_per_launch": ub,
             "bytes_definition": "unique HBM bytes per launch: the stored inverses (C n ld s), the index "
                                 "map (4 C n), the 32-column residual block once (packed BF16 hi/lo "
                                 "pairs, 128 N) and the FP32 local results (128 C n); the gathered "
                                 "residual rows that several cells share are counted once",
             "gathered_bytes_per_launch": fin["bytes"] / max(fin["launches"], 1)}
    return {"workload": describe(wl, sizes)["workload"], "dofs": sizes[-1]["n_dofs"], "nrhs": nrhs,
            "rhs": "b(U_j, nu) + c(w, w), U_j = linspace(0.2, 0.45, 32)", "rtol": args.rtol,
            "restart": args.multi_restart, "s_per_solve": ms / 1e3, "per_rhs_s": ms / 1e3 / nrhs,
            "iters": [i["iters"] for i in infos], "max_rel_res_true": max(i["rel_res_true"] for i in infos),
            "dtype": f"f64 Krylov/SpMM/coarse + {split_precision(prec)[0]} cell inverses "
                     f"({'tensor cores, ' if split_precision(prec)[0] == 'bf16' else ''}f32 accumulate); FP64 defects",
            "setup": {"build_hierarchy_s": build_s, "assemble_ms": e0.elapsed_time(e1), "factor_ms": e1.elapsed_time(e2)},
            "kernel_ms_per_solve_profiled": {k: v["ms"] for k, v in kern.items()},
            "finest_sweep": sweeps,
            "gpu_launches_per_solve": launches / steps,
            # the dominant kernel of this solve is the FP64 SpMM (most of its event time); the
            # multi-RHS Vanka products are reported beside it
            "roofline": spmm if spmm else vanka,
            "roofline_vanka_sweep": vanka,
            "cpu_baseline_note": "the FP64 oracle of this workload needs ~70 GB of host memory and hours; not timed"}


def gpu_leg_multi(args, local_rank):
    """Multi-RHS workload as the line's own workload (bench.py --workload c5_3d_k1)."""
    import torch

    from paper_2107_10561_gb300 import build as _build

    torch.cuda.set_device(local_rank)
    _build.build()
    prec = args.precisions.split(",")[-1]
    sampler = ClockSampler(local_rank)
    sampler.start()
    row = multi_row(args, args.workload, args.steps, args.warmup, split_precision(prec)[0])
    clocks = sampler.stop()
    line = {"metric": "GMG-GMRES s to 1e-8 rel. res (mixed vs FP64, one GB300); Vanka sweep GB/s",
            "value": row["s_per_solve"], "unit": "s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * row["s_per_solve"], "higher_is_better": False, "scaling": "weak",
            "vs_baseline": None, "dtype": row["dtype"], "data": "synthetic",
            "config": {"workload": row["workload"], "dofs": row["dofs"], "nrhs": row["nrhs"], "rhs": row["rhs"],
                       "rtol": args.rtol, "restart": row["restart"], "parallelism": "single GPU"},
            "gpu_launches": int(row["gpu_launches_per_solve"] * args.steps), "clocks": clocks,
            "roofline": row["roofline"], "multi": row, "cpu_baseline": None,
            "cpu_baseline_note": row["cpu_baseline_note"]}
    print(json.dumps(line))


def gpu_leg_newton(args, local_rank):
    """Damped Newton for the slab problem F(X) = A X + c(X, X) - b(U, nu) = 0 from the seeded state,
    U = 0.3; stop at 1e-10 or a reduction by 1e4 (Sec. 5.1). Each step re-assembles J on every level,
    factors every cell inverse and the coarse inverse, and solves with GMG-FGMRES to args.rtol."""
    import numpy as np
    import torch

    import synth
    from paper_2107_10561_gb300 import Hierarchy, make_params
    from paper_2107_10561_gb300 import build as _build

    torch.cuda.set_device(local_rank)
    _build.build()
    wl = workload(args.workload)
    out = {}
    for prec in args.precisions.split(","):
        p = hier_params(wl, prec, "additive")
        h = Hierarchy(p)
        idx = h.dof_lattice_index()
        X0 = torch.from_numpy(np.ascontiguousarray(synth.linearisation_point(wl).reshape(-1)[idx])).cuda()
        X = torch.empty_like(X0)
        for _ in range(args.warmup):
            X.copy_(X0)
            info = h.newton_solve(X, wl.inflow_u, rtol=args.rtol, restart=wl.restart)
        torch.cuda.synchronize()
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        launches0 = Hierarchy.kernel_launches()
        ev0.record()
        for _ in range(args.steps):
            X.copy_(X0)
            info = h.newton_solve(X, wl.inflow_u, rtol=args.rtol, restart=wl.restart)
        ev1.record()
        torch.cuda.synchronize()
        out[prec] = {"ms": ev0.elapsed_time(ev1) / args.steps, "info": info,
                     "launches": (Hierarchy.kernel_launches() - launches0) / args.steps}
        h.close()
    head = mode_precision(args)
    r = out[head]
    cfg = {"workload": f"{wl.name}: damped Newton for one slab, U = {wl.inflow_u}, from the seeded state",
           "stop": "||F|| <= max(1e-10, ||F_0|| / 1e4)", "linear_rtol": args.rtol, "parallelism": "single GPU"}
    line = {"metric": "damped-Newton slab solve s (GMG-FGMRES inner solves)", "value": r["ms"] / 1e3, "unit": "s",
            "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "ms_per_step": r["ms"],
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
            "dtype": dtype_label(head), "data": "synthetic", "config": cfg,
            "by_precision": {p: {"s": v["ms"] / 1e3, "newton_iters": v["info"]["newton_iters"],
                                 "gmres_iters": v["info"]["gmres_iters"], "res": v["info"]["res"],
                                 "lam": v["info"]["lam"]} for p, v in out.items()},
            "gpu_launches": int(r["launches"] * args.steps)}
    print(json.dumps(line))


def gpu_leg_march(args, local_rank):
    """Time marching (Problem 3.1): args.march slabs from the seeded state, slab n started from slab
    n-1 with its last time node as initial value, each solved by damped Newton (stop at 1e-10 or a
    reduction by 1e4) with GMG-FGMRES inner solves; the wake functional int_{I_n} int_wake v_1 per slab."""
    import numpy as np
    import torch

    import synth
    from paper_2107_10561_gb300 import Hierarchy, make_params
    from paper_2107_10561_gb300 import build as _build

    torch.cuda.set_device(local_rank)
    _build.build()
    wl = workload(args.workload)
    prec = mode_precision(args)
    p = hier_params(wl, prec, "additive")
    h = Hierarchy(p)
    idx = h.dof_lattice_index()
    X0 = torch.from_numpy(np.ascontiguousarray(synth.linearisation_point(wl).reshape(-1)[idx])).cuda()
    # wake: the two level-1 cell columns behind the obstacle at the obstacle's height (a full-height
    # box would measure the flux, which the inflow fixes)
    lo = (wl.obstacle_hi[0], wl.obstacle_lo[1]) + ((0,) if wl.dim == 3 else ())
    hi = (min(wl.obstacle_hi[0] + 2, wl.coarse_cells[0]), wl.obstacle_hi[1]) + \
        ((wl.coarse_cells[2],) if wl.dim == 3 else ())
    j = torch.empty(h.n_dofs(), dtype=torch.float64, device="cuda")
    h.functional_weights(lo, hi, j)
    h.time_march(X0, wl.inflow_u, 1, j=j, rtol=args.rtol, restart=wl.restart)  # warm-up slab
    torch.cuda.synchronize()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ev0.record()
    states, infos, values = h.time_march(X0, wl.inflow_u, args.march, j=j, rtol=args.rtol, restart=wl.restart)
    ev1.record()
    torch.cuda.synchronize()
    ms = ev0.elapsed_time(ev1)
    h.close()
    line = {"metric": "time-marching s per slab (damped Newton, GMG-FGMRES inner solves)",
            "value": ms / 1e3 / args.march, "unit": "s", "n_gpus": 1, "steps": args.march, "warmup": 1,
            "ms_per_step": ms / args.march, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
            "dtype": dtype_label(prec), "data": "synthetic",
            "config": {"workload": f"{wl.name}: {args.march} slabs of tau = {wl.tau} from the seeded state, "
                                   f"U = {wl.inflow_u}", "wake": {"lo": lo, "hi": hi}, "linear_rtol": args.rtol,
                       "parallelism": "single GPU"},
            "slabs": [{"newton_iters": i["newton_iters"], "gmres_step": i["gmres_step"], "res": i["res"],
                       "wake_functional": v} for i, v in zip(infos, values)]}
    print(json.dumps(line))


def gpu_leg_robustness(args, local_rank):
    """Sec. 5.3 / Table 5.4 on the synthetic channel: for nu in {1e-3, 5e-4, 3e-4, 2e-4, 1e-4} and
    omega_d in {1, 0.7}, one damped-Newton slab solve from the seeded state with V(4,4) cycles and
    tau = 0.005; reports Newton steps and FGMRES iterations per step (None: FGMRES did not reach the
    tolerance within 1000 iterations, the table's infinity)."""
    import dataclasses

    import numpy as np
    import torch

    import synth
    from paper_2107_10561_gb300 import Hierarchy, make_params
    from paper_2107_10561_gb300 import build as _build

    torch.cuda.set_device(local_rank)
    _build.build()
    base = workload(args.workload)
    prec = mode_precision(args)
    table = []
    t_all = time.perf_counter()
    for nu in (1e-3, 5e-4, 3e-4, 2e-4, 1e-4):
        for omega in (1.0, 0.7):
            wl = dataclasses.replace(base, nu=nu, omega=omega, nu1=4, nu2=4, tau=0.005)
            p = hier_params(wl, prec, "additive")
            h = Hierarchy(p)
            idx = h.dof_lattice_index()
            X = torch.from_numpy(np.ascontiguousarray(synth.linearisation_point(wl).reshape(-1)[idx])).cuda()
            t0 = time.perf_counter()
            info = h.newton_solve(X, wl.inflow_u, rtol=args.rtol, restart=wl.restart, max_iter=1000,
                                  raise_on_fail=False)
            torch.cuda.synchronize()
            dt = time.perf_counter() - t0
            ok = info["status"] == "STM_OK"
            table.append({"nu": nu, "omega_d": omega, "converged": ok, "newton_steps": info["newton_iters"],
                          "gmres_per_step": info["gmres_step"],
                          "gmres_avg": (float(np.mean(info["gmres_step"])) if ok and info["gmres_step"] else None),
                          "status": info["status"], "s": dt})
            h.close()
    line = {"metric": "Newton steps and FGMRES iterations per Newton step vs nu and omega_d (Table 5.4 setting)",
            "value": time.perf_counter() - t_all, "unit": "s", "n_gpus": 1, "steps": 1, "warmup": 0,
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": dtype_label(prec),
            "data": "synthetic",
            "config": {"workload": f"{base.name}, tau 0.005, V(4,4), additive Vanka, inner rtol {args.rtol}, "
                                   "FGMRES(30) capped at 1000 iterations", "parallelism": "single GPU"},
            "table": table}
    print(json.dumps(line))


def gpu_leg_mesh(args, local_rank):
    """Tables 5.1 and 5.5 setting on the synthetic channel: one linear FGMRES solve (seeded right-hand
    side, seeded linearisation point, rtol as given) with V(1,1) and with V(4,4) cycles while the same
    coarse grid is refined: 2D dG(1) on 3..6 levels, 3D dG(1) on 2..4 levels. The paper reports the
    average per Newton step over whole simulations; here each entry is one solve."""
    import dataclasses

    import numpy as np
    import torch

    import synth
    from paper_2107_10561_gb300 import Hierarchy
    from paper_2107_10561_gb300 import build as _build

    torch.cuda.set_device(local_rank)
    _build.build()
    prec = mode_precision(args)
    table = []
    t_all = time.perf_counter()
    for base_name, levels in (("c4_2d_k1", (3, 4, 5, 6)), ("c3_3d_k1", (2, 3, 4))):
        base = workload(base_name)
        for n_levels in levels:
            for sweeps in (1, 4):
                wl = dataclasses.replace(base, n_levels=n_levels, nu1=sweeps, nu2=sweeps)
                h = Hierarchy(hier_params(wl, prec, "additive"))
                idx = h.dof_lattice_index()
                X = torch.from_numpy(np.ascontiguousarray(synth.linearisation_point(wl).reshape(-1)[idx])).cuda()
                b = torch.from_numpy(np.ascontiguousarray(synth.random_rhs(wl).reshape(-1)[idx])).cuda()
                h.assemble_jacobian(X)
                h.factor_cells()
                x = torch.zeros_like(b)
                h.gmres_solve(b, x, rtol=args.rtol, restart=wl.restart, raise_on_fail=False)
                ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                x.zero_()
                torch.cuda.synchronize()
                ev0.record()
                info = h.gmres_solve(b, x, rtol=args.rtol, restart=wl.restart, raise_on_fail=False)
                ev1.record()
                torch.cuda.synchronize()
                table.append({"mesh": f"{wl.dim}D {'x'.join(map(str, wl.fine_cells))}", "levels": n_levels,
                              "dofs": h.n_dofs(), "cycle": f"V({sweeps},{sweeps})", "iters": info["iters"],
                              "converged": info["status"] == "STM_OK", "ms": ev0.elapsed_time(ev1)})
                h.close()
    line = {"metric": "FGMRES iterations per solve for V(1,1) / V(4,4) under refinement (Tables 5.1, 5.5 setting)",
            "value": time.perf_counter() - t_all, "unit": "s", "n_gpus": 1, "steps": 1, "warmup": 1,
            "higher_is_better": False, "scaling": "weak", "vs_baseline": None, "dtype": dtype_label(prec),
            "data": "synthetic",
            "config": {"workload": "2D channel 16x4 coarse cells (obstacle), dG(1), 3..6 levels; 3D channel "
                                   "16x4x4 coarse cells (obstacle), dG(1), 2..4 levels; additive Vanka, omega 0.7",
                       "rtol": args.rtol, "parallelism": "single GPU"},
            "table": table}
    print(json.dumps(line))


def reference_arm(args):
    """The CPU oracle on a bounded sample of the bench's workload (one refinement level fewer), each
    step one full oracle FGMRES solve, scaled to the full workload by the DoF ratio."""
    wl = workload(args.workload)
    if wl.extra.get("nrhs"):
        print(json.dumps({"impl": "reference", "unavailable": "the FP64 oracle of the 32-right-hand-side workload "
                                                              "needs ~70 GB of host memory and hours"}))
        return
    threads = os.cpu_count() or 1
    steps = max(1, min(args.steps, REFERENCE_MAX_STEPS))
    o = run_oracle(args.workload, args.rtol, steps, threads=threads, n_levels=sample_levels(wl))
    full_dofs = full_workload_dofs(wl)
    scale = full_dofs / o["sizes"]["n_dofs"]
    t = statistics.median(o["solve_s"]) * scale
    sample = (f"each step one full FP64 oracle FGMRES solve (rtol {args.rtol:g}) of the same 3D channel with one "
              f"refinement level fewer ({o['sizes']['n_levels']} levels, {o['sizes']['n_dofs']:,} DoFs, "
              f"{o['iters'][-1]} iterations), numpy/scipy with {threads} BLAS threads, after an untimed "
              f"{o['setup_s']:.1f} s oracle set-up; value = median step x {scale:.3f} (DoF ratio to the full "
              f"{full_dofs:,}-DoF workload); {steps} of the {args.steps} requested steps (at most "
              f"{REFERENCE_MAX_STEPS}, so that the run ends within a few minutes)")
    line = {"impl": "reference", "metric": "GMG-GMRES s to 1e-8 rel. res (mixed vs FP64, one GB300); Vanka sweep GB/s",
            "value": t, "unit": "s", "n_gpus": args.gpus, "steps": steps, "steps_requested": args.steps,
            "warmup": 0, "ms_per_step": 1e3 * t, "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
            "dtype": "f64", "data": "synthetic",
            "config": {"workload": describe(wl, [{"n_dofs": full_dofs, "n_cells": None, "n_local": None}])["workload"],
                       "dofs": full_dofs, "rtol": args.rtol, "parallelism": "CPU oracle (rank 0 of the job)"},
            "cpu_baseline": {"value": t, "unit": "s", "cores": threads, "kind": "oracle", "sample": sample,
                             "cpu_model": cpu_model()},
            "e2e": {"value": t, "unit": "s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))


def full_workload_dofs(wl):
    """DoFs of the finest level: (k+1)(d R + n_p C) from the node and cell counts of the obstacle
    channel (the same count the library reports)."""
    import numpy as np

    cells = wl.fine_cells
    f = 2 ** (wl.n_levels - 1)
    lo = [x * f for x in wl.obstacle_lo]
    hi = [x * f for x in wl.obstacle_hi]
    active = np.ones(cells[::-1], dtype=bool)  # (z,) y, x
    if any(h > l for l, h in zip(lo, hi)):
        sl = tuple(slice(l, h) for l, h in zip(lo[::-1], hi[::-1]))
        active[sl] = False
    nodes = np.zeros(tuple(2 * c + 1 for c in cells[::-1]), dtype=bool)
    for idx in zip(*np.nonzero(active)):
        nodes[tuple(slice(2 * i, 2 * i + 3) for i in idx)] = True
    C, R = int(active.sum()), int(nodes.sum())
    return (wl.k + 1) * (wl.dim * R + (wl.dim + 1) * C)


def kernel_driver(args):
    """Fixed launch sequences for ncu captures (one line of CUDA-event timings on stdout)."""
    import dataclasses

    import torch

    import synth
    from paper_2107_10561_gb300 import Hierarchy
    from paper_2107_10561_gb300 import build as _build

    torch.cuda.set_device(0)
    _build.build()
    wl = workload(args.workload)
    if args.levels:
        wl = dataclasses.replace(wl, n_levels=args.levels)
    prec = mode_precision(args)
    h = Hierarchy(hier_params(wl, prec, "additive"))
    h.assemble_jacobian(lattice_vec(h, synth.linearisation_point(wl)))
    h.factor_cells()
    g = h.finest
    n = h.n_dofs(g)
    gen = torch.Generator(device="cuda").manual_seed(7)
    out = {"driver": args.kernel_driver, "workload": wl.name, "levels": wl.n_levels, "precision": prec,
           "steps": args.steps}
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def timed(fn):
        fn()
        torch.cuda.synchronize()
        ev0.record()
        for _ in range(args.steps):
            fn()
        ev1.record()
        torch.cuda.synchronize()
        return 1e3 * ev0.elapsed_time(ev1) / args.steps

    if args.kernel_driver == "product_sweep":
        x = torch.randn(n, dtype=torch.float64, device="cuda", generator=gen)
        y, d = torch.empty_like(x), torch.zeros_like(x)
        out["product_us"] = timed(lambda: h.spmv(g, x, y))
        out["sweep_us"] = timed(lambda: h.vanka_sweep(g, x, d))
    elif args.kernel_driver in ("multi_sweep", "fused_sweep"):
        R = torch.randn(32, n, dtype=torch.float64, device="cuda", generator=gen)
        D = torch.zeros_like(R)
        fn = ((lambda: h.vanka_sweep_multi(g, R, D)) if args.kernel_driver == "multi_sweep"
              else (lambda: h.vanka_sweep_fused(g, R[:16], D[:16], R[16:], D[16:])))
        out["sweep_us"] = timed(fn)
        # the local products alone: event pairs around each launch inside the library
        h.profile_enable(True)
        for _ in range(args.steps):
            fn()
        loc = h.profile_read("vanka_local", g)
        h.profile_enable(False)
        out["local_us"] = 1e3 * loc["ms"] / max(loc["launches"], 1)
    else:
        n0 = h.n_dofs(0)
        r0 = torch.randn(n0, dtype=torch.float64, device="cuda", generator=gen)
        d0 = torch.empty_like(r0)
        out["coarse_us"] = timed(lambda: h.coarse_solve(r0, d0))
        out["coarse_transposed_us"] = timed(lambda: h.coarse_solve(r0, d0, transpose=True))
    out["sizes"] = h.sizes(g)
    h.close()
    print(json.dumps(out))


def main():
    args = parse()
    if args.kernel_driver:
        kernel_driver(args)
        return
    if args.oracle_child:
        oracle_child(args.oracle_child)
        return
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local_rank = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        if rank == 0:
            reference_arm(args)
        return

    if args.mesh_study:
        if rank == 0:
            gpu_leg_mesh(args, local_rank)
        return
    if args.newton:
        if rank == 0:
            gpu_leg_newton(args, local_rank)
        return
    if args.robustness:
        if rank == 0:
            gpu_leg_robustness(args, local_rank)
        return
    if args.march:
        if rank == 0:
            gpu_leg_march(args, local_rank)
        return
    if workload(args.workload).extra.get("nrhs"):
        if rank == 0:
            gpu_leg_multi(args, local_rank)
        return
    wl, sizes, results, errs, head, clocks, e2e_s, dist, fp64_peak, rows = gpu_leg(args, rank, world, local_rank)
    if rank != 0:
        if dist:
            dist.destroy_process_group()
        return
    precs = list(results)
    if not args.no_other_rows and world == 1:
        if args.workload != "c2_2d_k2":
            rows["c2_2d_k2"] = workload_row(args, "c2_2d_k2", [p for p in ("f64", "bf16", "bf16+f32d") if p in precs]
                                            or ["f64"], args.steps, args.warmup)
        rows["c5_3d_k1"] = multi_row(args, "c5_3d_k1", 1, 1)
    pk = peaks()
    hbm = pk["hbm_gbs"] if pk else 6800.0
    peak_src = "MEASURED_PEAKS.json hbm_gbs (of measured)" if pk else "fallback 6800 GB/s"
    r = results[head]
    vl = r["finest"]["vanka_local"]
    achieved = vl["bytes"] / (vl["ms"] * 1e-3) / 1e9 if vl["ms"] > 0 else None
    vk = "k_vanka_warp" if sizes[-1]["n_local"] <= 64 else "k_vanka_local"
    traffic = recorded_traffic(args.workload, vk, split_precision(head)[0])
    cfg = describe(wl, sizes)
    cfg["rtol"] = args.rtol
    inv_bytes = {"f64": 8, "f32": 4, "bf16": 2}
    cfg["l2"] = (f"inputs larger than L2: finest J {sizes[-1]['nnz'] * 12 / 1e6:.0f} MB, finest inverses "
                 f"{sizes[-1]['n_cells'] * sizes[-1]['n_local'] ** 2 * inv_bytes[split_precision(head)[0]] / 1e6:.0f} MB ({head})")
    cfg["parallelism"] = f"replicas x{world}" if world > 1 else "single GPU"
    line = {
        "metric": "GMG-GMRES s to 1e-8 rel. res (mixed vs FP64, one GB300); Vanka sweep GB/s",
        "value": r["ms_per_solve"] / 1e3, "unit": "s", "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": r["ms_per_solve"], "higher_is_better": False, "scaling": "weak", "vs_baseline": None,
        "dtype": dtype_label(head) + "; FP64 residual products in the V-cycle",
        "data": "synthetic", "config": cfg,
        "head_precision": head,
        "fp64_s": results["f64"]["ms_per_solve"] / 1e3 if "f64" in results else None,
        "speedup_vs_fp64": (results["f64"]["ms_per_solve"] / r["ms_per_solve"]) if "f64" in results else None,
        "error_reference": ("err_vs_fp64_solution: the FP64 GPU solution of the same system in the same run; "
                            "err_vs_oracle_sample: the FP64 oracle's solution of the bounded oracle sample"),
        "by_precision": by_precision_rows(results, errs, args.steps),
        "gpu_launches": int(r["launches_per_step"] * args.steps),
        "other_rows": rows,
        "roofline": None,
        "roofline_spmv_f64": spmv_roofline(r, wl, sizes, fp64_peak, args.workload, limb_hbm(wl, hbm), peak_src),
        "roofline_defect_f32": defect_roofline(results["bf16+f32d"], sizes, hbm, peak_src, args.workload)
        if "bf16+f32d" in results else None,
        "roofline_vanka_sweep": {"kernel": f"{vk} (y_T = J_T^{{-1}} t_T), finest level, {head} inverses",
                                 "bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s",
                                 "frac": (achieved / hbm) if achieved else None,
                                 "traffic": traffic["per_launch_bytes"] if traffic else None,
                                 "traffic_source": traffic["source"] if traffic else "no capture of the current kernel source",
                                 "all_levels_gbs": (r["kernels"]["vanka_local"]["bytes"] / (r["kernels"]["vanka_local"]["ms"] * 1e-3) / 1e9)
                                 if r["kernels"]["vanka_local"]["ms"] > 0 else None,
                                 "peak_source": peak_src,
                                 "bytes_per_launch": vl["bytes"] / max(vl["launches"], 1),
                                 "avg_launch_us": 1e3 * vl["ms"] / max(vl["launches"], 1)},
        "vanka_sweep_gbs": achieved,
        "clocks": clocks,
        "e2e": {"value": e2e_s, "unit": "s", "h2d_bytes_per_step": sizes[-1]["n_dofs"] * 8,
                "d2h_bytes_per_step": sizes[-1]["n_dofs"] * 8,
                "path": f"stm_gmres_solve_host ({head}), pinned host b and x"},
    }
    # the dominant kernel of the head run: the finest-level class with the most event time per solve
    shares = {"roofline_vanka_sweep": r["finest"]["vanka_local"]["ms"],
              "roofline_spmv_f64": r["finest"]["jacobian_spmv"]["ms"]}
    dom = max((k for k in shares if line[k]), key=lambda k: shares[k])
    line["roofline"] = dict(line[dom], dominant_of={k: round(v / args.steps, 3) for k, v in shares.items()},
                            dominant_of_unit="ms per solve, finest level, profiled pass")
    if not args.no_cpu_baseline and world == 1:
        try:
            x_out = os.path.join(tempfile.mkdtemp(prefix="stm_xo_"), "x_oracle.npy")
            nl = sample_levels(wl)
            # the two thread counts run side by side on disjoint cores: one core for the 1-thread run,
            # the others for the all-thread run (when the host has more than one core)
            ncpu = os.cpu_count() or 1
            split = ncpu > 1 and hasattr(os, "sched_setaffinity")
            h1 = start_oracle(args.workload, args.rtol, 3, sweeps=3, n_levels=nl, threads=1, x_out=x_out,
                              cpus=[0] if split else None)
            if not split:
                o1 = finish_oracle(h1)
            hn = start_oracle(args.workload, args.rtol, 3, sweeps=3, n_levels=nl, threads=max(1, ncpu - 1),
                              cpus=list(range(1, ncpu)) if split else None)
            if split:
                o1 = finish_oracle(h1)
            on = finish_oracle(hn)
            line["cpu_baseline"] = cpu_baseline_entry(o1, on, sizes[-1]["n_dofs"], sizes[-1]["n_cells"],
                                                      r["iters_timed"], wl)
            import numpy as np

            chk = oracle_sample_check(args, wl, precs, np.load(x_out))
            for p, e in chk.items():
                line["by_precision"][p]["err_vs_oracle_sample"] = e
            line["oracle_sample_iters"] = o1["iters"][-1]
        except Exception as e:  # reported, never silently replaced
            line["cpu_baseline"] = {"value": None, "error": str(e)[-300:]}
    print(json.dumps(line))
    if dist:
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
