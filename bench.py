#!/usr/bin/env python
"""Benchmark of the FMM-BEM preconditioner (arXiv:1308.3339) on GB300.

Workload (default): 2-D Poisson -lap u = f on the unit square, 5-point FD on a 1024 x 1024
interior grid (N = 1,048,576), f a seeded mixture of 16 Gaussians, preconditioner =
FP32 FMM (p = 10, leaf 8x8, theta = 0.4) plus the boundary-element correction, FP64 FGMRES.

One step = one preconditioner apply z = P^{-1} r (all FMM + boundary stages).  The line
reports FMM apply points/s (N / apply time, L2 flushed between timed applies), the same
through the C ABI with host buffers (e2e), time-to-solution at relative residual 1e-8 for
the mixed (FP32 FMM, FP64 Krylov) and plain FP64 forms, the roofline of the dominant
kernel, and the CPU oracle timed on this host.  Multi-GPU: one independent problem per
rank (weak scaling, no collective in the data path).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = ("FMM apply points/sec and time-to-solution at rel. residual 1e-8, mixed vs plain "
          "on 1 GB300")
UNIT = "points/s"
SMS, LANES, SM_MAX_MHZ = 152, 128, 2070.0  # GB300: SMs, FP32 lanes per SM, max SM clock
FORMS = {"mixed_bf16": "FP32 P2P (3xFP16 tensor cores, per-leaf scales) and expansions, BF16 tensor-core M2L",
         "mixed_tf32": "FP32 P2P (3xFP16 tensor cores, per-leaf scales) and expansions, TF32 tensor-core M2L",
         "fp32": "FP32 FMM, CUDA-core M2L", "fp64": "FP64 FMM on CUDA cores"}
DTYPES = {"mixed_bf16": "f32+bf16", "mixed_tf32": "f32+tf32", "fp32": "f32", "fp64": "f64"}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--side", dest="n", type=int, default=1024, help="interior grid side n")
    ap.add_argument("--p", type=int, default=10)
    ap.add_argument("--leaf", type=int, default=64)
    ap.add_argument("--theta", type=float, default=0.4)
    ap.add_argument("--precision", default="mixed_tf32", choices=["mixed_bf16", "mixed_tf32", "fp32", "fp64"],
                    help="FMM form of the headline apply (FP64 Krylov in every form)")
    ap.add_argument("--no-tts", action="store_true", help="skip time-to-solution runs")
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU oracle baseline")
    ap.add_argument("--oracle-legs", action="store_true",
                    help="also time the FP64 oracle on the 64^2, 2048^2, 4096^2 and batched workloads (minutes)")
    ap.add_argument("--p2p", choices=["tc", "simt"], default="tc",
                    help="near-field engine of the headline apply (tensor cores or CUDA cores)")
    ap.add_argument("--solve-mode", choices=["graph", "host"], default="graph",
                    help="time-to-solution solves as one CUDA graph, or driven by the host "
                         "(kernel by kernel, as a profiler can see them)")
    ap.add_argument("--tts-forms", default="mixed_tf32,mixed_bf16,fp32,fp64",
                    help="precision forms whose time to solution is measured (comma list)")
    ap.add_argument("--configs", default="c1,c3,c4,c5",
                    help="further workloads timed after the headline (comma list of c1,c3,c4,c5; '' for none)")
    a = ap.parse_args()
    a.configs = [c for c in a.configs.split(",") if c]
    a.tts_forms = [f for f in a.tts_forms.split(",") if f]
    return a


def workload(args):
    return {"workload": f"poisson-fd {args.n}x{args.n} gaussian-mixture(16) FMM-BEM precond",
            "n": args.n, "N": args.n * args.n, "p": args.p, "leaf_max": args.leaf,
            "theta": args.theta, "krylov": "FGMRES(30) FP64", "fmm": FORMS[args.precision],
            "p2p_engine": "tensor cores" if args.p2p == "tc" else "CUDA cores",
            "l2": "flushed: 256 MB write between timed applies"}


# ---------------------------------------------------------------- clocks
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.idx = gpu_index
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.idx), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "20"], stdout=self.fh,
                stderr=subprocess.DEVNULL)
        except (FileNotFoundError, OSError):
            self.proc = None
            return
        # the timed region starts once the sampler is producing lines (at most ~3 s)
        for _ in range(300):
            if self.proc.poll() is not None or os.path.getsize(self.path) > 0:
                break
            time.sleep(0.01)

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.fh.close()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        os.unlink(self.path)
        return {"sm_mhz": float(np.median(sm)) if sm else None,
                "sm_max_mhz": float(max(smax)) if smax else None,
                "samples": len(sm), "reasons": sorted(reasons)}


# ---------------------------------------------------------------- distributed
def dist_setup():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    pg = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl" if os.environ.get("FMMPC_BENCH_BACKEND", "nccl") == "nccl" else "gloo")
        pg = dist
    return world, rank, local, pg


def max_over_ranks(x: float, pg, device) -> float:
    if pg is None:
        return x
    import torch
    t = torch.tensor([x], dtype=torch.float64, device=device)
    pg.all_reduce(t, op=pg.ReduceOp.MAX)
    return float(t.item())


def barrier(pg):
    if pg is not None:
        pg.barrier()


# ---------------------------------------------------------------- CPU oracle
def cpu_baseline(args, repeats=1):
    import oracle as O
    import synth_inputs as S
    n = args.n
    f = S.gaussian_mixture(n, 0)
    t0 = time.perf_counter()
    Pr = O.Problem(n, p=args.p, leaf_max=args.leaf, theta=(int(round(args.theta * 1000)), 1000))
    t_setup = time.perf_counter() - t0
    ts = []
    for _ in range(repeats):
        t0 = time.perf_counter()
        Pr.apply(f, "fmm")
        ts.append(time.perf_counter() - t0)
    t = float(np.mean(ts))
    return {"value": n * n / t, "unit": UNIT, "cores": O.threads(), "kind": "oracle",
            "sample": f"{repeats} full FP64 FMM-BEM apply of the {n}x{n} workload (setup {t_setup:.1f} s excluded)",
            "seconds_per_apply": t}


def oracle_legs(args):
    """The FP64 oracle on the host cores for the other workloads, one right-hand side each,
    not extrapolated: c1 a full GMRES(30) solve at 64^2; c3 one apply at 4096^2; c5 one
    apply and one FGMRES(30) solve at 2048^2; c4 one apply and one solve of a stated subset
    of the 64 problems (one of each side 128 .. 1024).  Set-up (tree, lists, the dense
    BEM LU) is reported apart.  Opt-in (--oracle-legs): the 4096^2 LU alone takes minutes."""
    import oracle as O
    import synth_inputs as S
    out = {"cores": O.threads()}

    def leg(n, f, solve, method="fgmres"):
        t0 = time.perf_counter()
        R = O.Problem(n, p=10)
        rec = {"n": n, "setup_s": time.perf_counter() - t0}
        t0 = time.perf_counter()
        R.apply(f, "fmm")
        rec["apply_s"] = time.perf_counter() - t0
        rec["apply_points_per_s"] = n * n / rec["apply_s"]
        if solve:
            t0 = time.perf_counter()
            _, it, rr, conv = R.solve(f, method, 30, 200, 1e-8, "fmm")
            rec.update(solve_s=time.perf_counter() - t0, iters=it, rel_res=rr, converged=bool(conv))
        return rec

    f1, _ = S.manufactured_sin(64)
    t0 = time.perf_counter()
    R = O.Problem(64, p=8)
    _, it, rr, _ = R.solve(f1, "gmres", 30, 200, 1e-8, "fmm")
    out["c1"] = {"n": 64, "solve_s": time.perf_counter() - t0, "iters": it, "rel_res": rr, "note": "set-up included"}
    sides = [int(v) for v in S.batched_sides(0, 64)]
    subset = [sides.index(n) for n in (128, 256, 512, 1024) if n in sides]
    out["c4_subset"] = [dict(problem=k, **leg(sides[k], S.gaussian_mixture(sides[k], 1000 + k), True)) for k in subset]
    out["c5"] = leg(2048, S.gaussian_mixture(2048, 3), True)
    out["c3"] = leg(4096, S.gaussian_mixture(4096, 0), False)
    return out


def run_reference(args):
    world, rank, local, pg = dist_setup()
    if rank != 0:
        return
    import oracle as O
    import synth_inputs as S
    n = args.n
    f = S.gaussian_mixture(n, 0)
    Pr = O.Problem(n, p=args.p, leaf_max=args.leaf, theta=(int(round(args.theta * 1000)), 1000))
    for _ in range(args.warmup):
        Pr.apply(f, "fmm")
    t0 = time.perf_counter()
    for _ in range(args.steps):
        Pr.apply(f, "fmm")
    t = (time.perf_counter() - t0) / args.steps
    v = n * n / t
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": t * 1e3,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": workload(args),
            "cpu_baseline": {"value": v, "unit": UNIT, "cores": O.threads(), "kind": "oracle",
                             "sample": f"one full FP64 FMM-BEM apply of the {n}x{n} workload per step"},
            "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------- GPU arm
def traffic_record(kernel: str):
    """DRAM bytes per launch of a kernel from the committed ncu summary, valid only while
    the kernel's source file is unchanged (its hash is stored beside the figure)."""
    path = os.path.join(ROOT, "profiles", "traffic.json")
    try:
        rec = json.load(open(path))[kernel]
        src = os.path.join(ROOT, "paper_1308_3339_gb300", "csrc", rec["source"])
        h = hashlib.sha256(open(src, "rb").read()).hexdigest()[:16]
        if rec.get("source_sha256_16") == h:
            return rec
    except (OSError, ValueError, KeyError):
        pass
    return None


def load_peaks():
    try:
        return json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except (OSError, ValueError):
        return None


def rooflines(P, stage_ms, nrhs=1):
    """Roofline of the P2P and M2L kernels of the handle's form from their live CUDA-event
    times; the dominant one (larger time) is reported as `roofline`."""
    m = P.query("leaf_side")
    digits = P.precision == "fp64"  # tensor cores: 28 products of FP16 digits per FP64 product
    pk = load_peaks()
    out = {}
    # P2P: one FMA (2 flops) per source-target pair of the near-field lists
    pairs = P.query("n_p2p") * m ** 4 * nrhs
    t = stage_ms["p2p"]
    if P.query("tc_p2p"):
        # FP16 operands: the dense FP16 rate is the BF16 rate
        if pk:
            peak, src = pk["bf16_tflops"], f"measured bf16 burst {pk['bf16_tflops']:.1f} TFLOP/s (FP16 runs at the BF16 rate)"
        else:
            peak, src = 1900.0, "fallback bf16 1.9 PFLOP/s (FP16 runs at the BF16 rate)"
        ach = 2.0 * pairs / (t * 1e-3) / 1e12
        mult = 28 if digits else 3
        how = ("each FP64-accurate product takes 28 FP16 MMAs (pairs of 9-bit digits)" if digits else
               "each FP32-accurate product takes 3 FP16 MMAs (hi*hi, hi*lo, lo*hi)")
        out["p2p"] = {"bound": "tensor",
                      "kernel": "k_p2p_oz (lattice P2P, tcgen05 FP16 digits)" if digits else
                                "k_p2p_tc (lattice P2P, tcgen05 FP16 x3)",
                      "achieved": ach, "peak": peak, "unit": "TFLOP/s",
                      "peak_source": f"{src}; {how}, so the tensor pipe executes {mult}x the algorithmic flops",
                      "executed_frac": mult * ach / peak,
                      "work": f"{pairs:.4e} pairs/launch x 2 flop", "launch_ms": t}
    else:
        peak = SMS * LANES * 2 * SM_MAX_MHZ * 1e6 / 1e12
        out["p2p"] = {"bound": "alu", "kernel": "k_p2p (lattice P2P, CUDA cores)",
                      "achieved": 2.0 * pairs / (t * 1e-3) / 1e12, "peak": peak, "unit": "TFLOP/s",
                      "peak_source": f"FP32 FMA lanes {SMS}x{LANES} x 2 flop x {SM_MAX_MHZ:.0f} MHz max SM clock",
                      "work": f"{pairs:.4e} pairs/launch x 2 flop", "launch_ms": t}
    # M2L: 8 p^2 real flops per (target, source) pair
    p = P.p
    t = stage_ms["m2l"]
    tcm = P.query("tc_m2l")
    if digits and p <= 15:
        pairs_m = P.query("n_m2l") * nrhs
        peak = pk["bf16_tflops"] if pk else 1900.0
        out["m2l"] = {"bound": "tensor", "kernel": "k_m2l_oz (+ k_m2l_oz_pack, k_m2l_oz_sum; tcgen05 FP16 digits)",
                      "achieved": 8.0 * p * p * pairs_m / (t * 1e-3) / 1e12, "peak": peak, "unit": "TFLOP/s",
                      "peak_source": ("measured bf16 burst" if pk else "fallback bf16") + ", 28 digit products each",
                      "work": f"{pairs_m} pairs/launch x 8p^2 flop (p={p})", "launch_ms": t}
    elif tcm:
        pairs_m = P.query("n_m2l") * nrhs  # volume pairs; boundary sources run in stage m2l_bnd
        if tcm == 2:
            peak = pk["bf16_tflops"] if pk else 1900.0
            src = "measured bf16 burst" if pk else "fallback bf16 1.9 PFLOP/s"
        else:
            peak = (pk["bf16_tflops"] if pk else 1900.0) * 1.1 / 2.25
            src = "measured bf16 burst x nominal TF32/BF16 ratio 1.1/2.25" if pk else "fallback bf16 x 1.1/2.25"
        out["m2l"] = {"bound": "tensor", "kernel": "k_m2l_tc (+ k_m2l_pack, operand images)",
                      "achieved": 8.0 * p * p * pairs_m / (t * 1e-3) / 1e12, "peak": peak, "unit": "TFLOP/s",
                      "peak_source": src, "work": f"{pairs_m} pairs/launch x 8p^2 flop (p={p})", "launch_ms": t}
    else:
        m2l_pairs = (P.query("n_m2l") + P.query("n_m2l_vb")) * nrhs
        peak = SMS * LANES * 2 * SM_MAX_MHZ * 1e6 / 1e12
        out["m2l"] = {"bound": "alu", "kernel": "k_m2l_vol (+ k_root_const, 1 block)",
                      "achieved": 8.0 * p * p * m2l_pairs / (t * 1e-3) / 1e12, "peak": peak, "unit": "TFLOP/s",
                      "peak_source": f"FP32 FMA lanes {SMS}x{LANES} x 2 flop x {SM_MAX_MHZ:.0f} MHz max SM clock",
                      "work": f"{m2l_pairs} pairs/launch x 8p^2 flop (p={p})", "launch_ms": t}
    for k, v in out.items():
        v["frac"] = v["achieved"] / v["peak"]
        rec = traffic_record(v["kernel"].split()[0])
        v["traffic"] = rec["bytes_per_launch"] if rec else None
    dom = max(out, key=lambda k: out[k]["launch_ms"])
    return out[dom], out


def time_solves(P, fd, reps, rtol=1e-8, graphs=2, **kw):
    """Median wall time of P.solve (host clock around the call, device synchronised on
    both sides: the solve returns after its convergence test) after one warm-up solve."""
    import torch
    P.solve(fd, rtol=rtol, use_graphs=graphs, **kw)  # warm-up (workspace, graphs)
    out = []
    for _ in range(reps):
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        u, info = P.solve(fd, rtol=rtol, use_graphs=graphs, **kw)
        torch.cuda.synchronize()
        out.append((time.perf_counter() - t0) * 1e3)
        last = info
    return {"ms": float(np.median(out)), "iters": last["iters"], "rel_res": last["rel_res"],
            "status": last["status"], "mode": {0: "host loop", 1: "host loop + apply graphs",
                                                2: "one graph (device-side convergence)"}[graphs]}


def time_apply(P, r, z, flush, reps=10):
    """Mean CUDA-event time of one apply (L2 flushed before each) on the current stream."""
    import torch
    stream = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    ts = []
    for i in range(reps + 3):
        flush.zero_()
        e0.record(stream)
        P.apply(r, out=z)
        e1.record(stream)
        e1.synchronize()
        if i >= 3:
            ts.append(e0.elapsed_time(e1))
    return float(np.mean(ts))


def bench_c1(args, flush):
    """64 x 64, manufactured sin solution, p = 8, GMRES(30) to 1e-8 (FGMRES in the single-
    precision forms, whose preconditioner is not exactly linear)."""
    import torch
    import synth_inputs as S
    from paper_1308_3339_gb300 import FmmPreconditioner
    n = 64
    f, _ = S.manufactured_sin(n)
    fd = torch.tensor(f, dtype=torch.float64, device="cuda")
    out = {}
    for form in ("mixed_tf32", "fp32", "fp64"):
        P = FmmPreconditioner(n, p=8, precision=form)
        method = "gmres" if form == "fp64" else "fgmres"
        out[form] = {"method": method, "apply_ms": time_apply(P, fd, torch.empty_like(fd), flush),
                     **time_solves(P, fd, 5, method=method)}
        P.close()
    return {"workload": "poisson-fd 64x64 manufactured sin, p=8, leaf 8x8, theta 0.4", **out}


def bench_c3(args, flush):
    """4096 x 4096 x 32 right-hand sides, p = 10: apply points/s (N R / t), FGMRES(15) and
    PCG time to 1e-8 in the mixed TF32 and plain FP32 forms; M2L roofline of the 32-RHS apply."""
    import torch
    import synth_inputs as S
    from paper_1308_3339_gb300 import FmmPreconditioner
    n, R = 4096, 32
    rs = torch.tensor(np.stack([S.gaussian_mixture(n, k) for k in range(R)]), dtype=torch.float64, device="cuda")
    z = torch.empty_like(rs)
    out = {"workload": "poisson-fd 4096x4096 x 32 rhs gaussian-mixture(16), p=10, FGMRES(15) to 1e-8"}
    for form in ("mixed_tf32", "fp32"):
        t0 = time.perf_counter()
        P = FmmPreconditioner(n, p=10, precision=form, n_rhs=R)
        torch.cuda.synchronize()
        setup_ms = (time.perf_counter() - t0) * 1e3
        ta = time_apply(P, rs, z, flush, reps=5)
        P.set_timing(2)
        P.apply(rs, out=z)
        st = P.stage_times()
        P.set_timing(0)
        _, allr = rooflines(P, st, nrhs=R)
        rec = {"setup_ms": setup_ms, "apply_ms": ta, "points_per_s": n * n * R / (ta * 1e-3)}
        for k in ("m2l", "p2p"):
            rec[f"{k}_roofline"] = {q: allr[k][q] for q in ("kernel", "achieved", "peak", "unit", "frac", "launch_ms",
                                                            "work")}
        rec.update(time_solves(P, rs, 1, restart=15))
        # preconditioned CG on the same 32 right-hand sides: the short recurrence keeps the
        # FP64 vector work per iteration (the FP64 pipe's share of the step) small
        rec["pcg"] = time_solves(P, rs, 1, method="cg")
        out[form] = rec
        P.close()
        torch.cuda.empty_cache()
    return out


def bench_c4(args, flush):
    """64 problems of sides drawn from {128, ..., 2048} (seed 0), each its own Gaussian
    mixture (seed 1000 + k): one graph solving all of them side by side (FGMRES(30) to
    1e-8) against the sum of the same problems solved one at a time."""
    import torch
    import synth_inputs as S
    from paper_1308_3339_gb300 import FmmBatch, FmmPreconditioner
    sides = [int(v) for v in S.batched_sides(0, 64)]
    fs = [torch.tensor(S.gaussian_mixture(n, 1000 + k), dtype=torch.float64, device="cuda")
          for k, n in enumerate(sides)]
    out = {"workload": "64 poisson-fd problems, sides from {128,256,512,1024,2048} (seed 0), p=10",
           "nodes": int(sum(n * n for n in sides))}
    for form in ("mixed_tf32", "fp32"):
        t0 = time.perf_counter()
        B = FmmBatch(sides, p=10, precision=form)
        torch.cuda.synchronize()
        setup_ms = (time.perf_counter() - t0) * 1e3
        B.solve(fs, rtol=1e-8)  # warm-up: workspace and the batch graph
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        us, infos = B.solve(fs, rtol=1e-8)
        torch.cuda.synchronize()
        t_batch = (time.perf_counter() - t0) * 1e3
        B.close()
        t_single = 0.0
        for k, n in enumerate(sides):
            P = FmmPreconditioner(n, p=10, precision=form)
            P.solve(fs[k], rtol=1e-8)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            P.solve(fs[k], rtol=1e-8)
            torch.cuda.synchronize()
            t_single += (time.perf_counter() - t0) * 1e3
            P.close()
        out[form] = {"setup_ms": setup_ms, "batched_ms": t_batch, "sum_single_ms": t_single,
                     "speedup": t_single / t_batch, "max_iters": max(i["iters"] for i in infos),
                     "all_converged": all(i["status"] == 0 for i in infos)}
        torch.cuda.empty_cache()
    return out


def bench_c5(args, flush):
    """Source inversion at 2048 x 2048: gradient of ||u(f) - u_obs||^2 through the adjoint
    FMM-preconditioned solve (forward + backward time), and a central-difference check of
    the gradient along one random direction (GPU only)."""
    import torch
    import synth_inputs as S
    from paper_1308_3339_gb300 import FmmPreconditioner
    from paper_1308_3339_gb300.autograd import fmm_solve
    n = 2048
    P = FmmPreconditioner(n, p=10, precision="mixed_tf32")
    f_true = torch.tensor(S.gaussian_mixture(n, 3), dtype=torch.float64, device="cuda")
    u_true, _ = P.solve(f_true, rtol=1e-10)
    noise = torch.tensor(np.random.default_rng(7).normal(0.0, 0.01, n * n), device="cuda")
    u_obs = u_true + noise
    f0 = torch.zeros(n * n, dtype=torch.float64, device="cuda", requires_grad=True)

    def loss(f):
        return ((fmm_solve(f, P, rtol=1e-10) - u_obs) ** 2).sum()

    loss(f0).backward()  # warm-up
    f0.grad = None
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    L = loss(f0)
    torch.cuda.synchronize()
    t_fwd = (time.perf_counter() - t0) * 1e3
    t0 = time.perf_counter()
    L.backward()
    torch.cuda.synchronize()
    t_bwd = (time.perf_counter() - t0) * 1e3
    g = f0.grad.detach()
    # the same at a non-zero iterate (f = f_true / 2), where the forward solve has work to do
    f1 = (0.5 * f_true).clone().requires_grad_(True)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    L1 = loss(f1)
    torch.cuda.synchronize()
    t_fwd1 = (time.perf_counter() - t0) * 1e3
    t0 = time.perf_counter()
    L1.backward()
    torch.cuda.synchronize()
    t_bwd1 = (time.perf_counter() - t0) * 1e3
    d = torch.tensor(np.random.default_rng(1).standard_normal(n * n), device="cuda")
    d /= d.norm()
    delta = 1e-2
    with torch.no_grad():
        fd = (loss(f0 + delta * d) - loss(f0 - delta * d)).item() / (2 * delta)
    gd = float(g @ d)
    P.close()
    return {"workload": "source inversion 2048x2048, loss ||u(f)-u_obs||^2, f0 = 0, mixed TF32, rtol 1e-10",
            "forward_ms": t_fwd, "backward_ms": t_bwd, "at_half_f_true": {"forward_ms": t_fwd1, "backward_ms": t_bwd1},
            "fd_check": {"directional_grad": gd, "central_difference": fd,
                         "rel_err": abs(fd - gd) / max(abs(fd), 1e-300)}}


def run_ours(args):
    import torch

    world, rank, local, pg = dist_setup()
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    import synth_inputs as S
    from paper_1308_3339_gb300 import FmmPreconditioner, _lib

    n = args.n
    N = n * n
    f = S.gaussian_mixture(n, rank)
    P = FmmPreconditioner(n, p=args.p, leaf_max=args.leaf, theta=args.theta, precision=args.precision)
    P.set_p2p_engine(args.p2p)
    r = torch.tensor(f, dtype=torch.float64, device=dev)
    z = torch.empty_like(r)
    flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=dev)  # 256 MB > L2
    stream = torch.cuda.current_stream()
    # warm-up of all three timing modes (each keeps its own captured graph)
    for mode in (0, 2, 1):
        P.set_timing(mode)
        for _ in range(max(args.warmup, 3)):
            P.apply(r, out=z)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)

    def timed(steps, mode):
        """Flush L2, apply, per step; events on the launching stream around each apply."""
        P.set_timing(mode)
        ts, st = [], {}
        for _ in range(steps):
            flush.zero_()
            e0.record(stream)
            P.apply(r, out=z)
            e1.record(stream)
            e1.synchronize()
            ts.append(e0.elapsed_time(e1))
            if mode:
                for k, v in P.stage_times().items():
                    st[k] = st.get(k, 0.0) + v / steps
        return ts, st

    # A: the headline, no stage events inside the apply
    barrier(pg)
    clocks = ClockSampler(local)
    clocks.start()
    t_wall0 = time.perf_counter()
    times, _ = timed(args.steps, 0)
    torch.cuda.synchronize()
    barrier(pg)
    wall = time.perf_counter() - t_wall0
    launches = P.query("launches")
    t_apply = float(np.mean(times))
    t_apply_max = max_over_ranks(t_apply, pg, dev)
    value = world * N / (t_apply_max * 1e-3)
    # B: the roofline kernels, timed live with events around the M2L and P2P kernels only
    tb, roof_ms = timed(args.steps, 2)
    # C: every stage (eleven event records; the breakdown, not the headline)
    _, stage_ms = timed(min(args.steps, 30), 1)
    P.set_timing(0)
    torch.cuda.synchronize()
    clk = clocks.stop()  # sampled over the three timed regions

    roofline, all_rooflines = rooflines(P, roof_ms)
    roofline["region_ms_per_step"] = float(np.mean(tb))

    # end to end through the C ABI with pinned host buffers
    rh = torch.tensor(f, dtype=torch.float64).pin_memory()
    zh = torch.empty_like(rh).pin_memory()
    lib = _lib.load()
    import ctypes as C
    for _ in range(2):
        _lib.check(lib.fmmpc_apply_host(P._h, C.c_void_p(rh.data_ptr()), C.c_void_p(zh.data_ptr()), 1), P._h)
    te = []
    for _ in range(max(3, args.steps // 2)):
        flush.zero_()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        _lib.check(lib.fmmpc_apply_host(P._h, C.c_void_p(rh.data_ptr()), C.c_void_p(zh.data_ptr()), 1), P._h)
        te.append(time.perf_counter() - t0)
    t_e2e = max_over_ranks(float(np.mean(te)), pg, dev)
    e2e = {"value": world * N / t_e2e, "unit": UNIT, "h2d_bytes_per_step": 8 * N, "d2h_bytes_per_step": 8 * N}

    tts = None
    if not args.no_tts:
        # every form timed the same way: applies replayed from their graphs, solves as one
        # graph each, so the forms differ only in their arithmetic
        P.set_timing(False)
        tts = {}
        for form in ("mixed_tf32", "mixed_bf16", "fp32", "fp64"):
            if form not in args.tts_forms:
                continue
            t0 = time.perf_counter()
            Pf = P if form == args.precision else FmmPreconditioner(n, p=args.p, leaf_max=args.leaf,
                                                                     theta=args.theta, precision=form)
            torch.cuda.synchronize()
            setup_ms = (time.perf_counter() - t0) * 1e3 if Pf is not P else None
            Pf.set_graphs(True)
            mode = 2 if args.solve_mode == "graph" else 0
            tts[form] = {"apply_ms": time_apply(Pf, r, z, flush),
                         **time_solves(Pf, r, 3 if form != "fp64" else 2, graphs=mode)}
            # preconditioned CG, the paper's own Krylov method (Sec. 6): a short recurrence,
            # so far fewer FP64 vector operations per iteration than FGMRES's CGS2
            tts[form]["pcg"] = time_solves(Pf, r, 3 if form != "fp64" else 2, graphs=mode, method="cg")
            _, inf = Pf.solve(r, rtol=1e-8)
            tts[form]["t_setup_ms"] = inf["t_setup_ms"]
            if form == args.precision:
                tts[form]["host_loop"] = time_solves(Pf, r, 3, graphs=1)
                tts[form]["solve_over_iters_x_apply"] = tts[form]["ms"] / (tts[form]["iters"] * tts[form]["apply_ms"])
            if Pf is not P:
                Pf.close()

    configs = {}
    for name, fn in (("c1", bench_c1), ("c3", bench_c3), ("c4", bench_c4), ("c5", bench_c5)):
        if name in args.configs and world == 1:
            t0 = time.perf_counter()
            try:
                configs[name] = fn(args, flush)
            except Exception as e:  # reported, not hidden: the line says which config failed
                import traceback
                configs[name] = {"error": f"{type(e).__name__}: {e}",
                                 "where": traceback.format_exc().strip().splitlines()[-6:]}
            configs[name]["bench_wall_s"] = time.perf_counter() - t0
            torch.cuda.empty_cache()

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu:
        cpu = cpu_baseline(args)
        if args.oracle_legs:
            cpu["other_workloads"] = oracle_legs(args)

    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": t_apply_max, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": DTYPES[args.precision], "data": "synthetic",
                "config": workload(args), "clocks": clk, "e2e": e2e,
                "gpu_launches": int(launches * args.steps), "roofline": roofline, "rooflines": all_rooflines,
                "cpu_baseline": cpu,
                "time_to_solution": tts, "stage_ms": stage_ms, "timed_wall_s": wall, "configs": configs}
        print(json.dumps(line), flush=True)
    if pg is not None:
        pg.destroy_process_group()


def main():
    args = parse()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
