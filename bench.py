#!/usr/bin/env python3
"""Benchmark of the pairing-Hamiltonian ground-state solver on one GB300.

Workload (default): Omega = 24 orbits, N = 12 pairs, dim C(24,12) = 2,704,156,
e ~ sorted U[-10,10], G_ij = -g_i g_j + eta_ij (seed 1).  One step = one full
ground-state solve in the chosen form (FP32-vector mixed precision with FP64
dots, FP64 tridiagonal solve and FP64 Rayleigh refinement; random start),
inputs resident on the device, L2 flushed between steps.

value = H*x off-diagonal nonzeros processed per second over the timed solves
(the paper's nonzero count C(Omega,N) N (Omega-N) per product, Sec. 5.3);
time-to-E0 of the chosen form and of plain FP64 Lanczos are reported beside it.

--impl reference times the CPU oracle (the plain FP64 program in oracle/) on
bounded row samples of the same H*x, in the same unit.
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
from pathlib import Path

import numpy as np

ROOT = Path(__file__).resolve().parent
sys.path.insert(0, str(ROOT))

import pd_inputs  # noqa: E402

WORKLOAD = "omega24_n12_sepnoise_s1"
METRIC = "H*x nonzeros/s over a full ground-state solve (time-to-E0 at rel err 1e-8: mixed form vs plain FP64 Lanczos)"
UNIT = "nnz/s"
L2_FLUSH_BYTES = 512 << 20       # > 129 MB L2


def parse_args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=None,
                    help="timed steps (default: 30 for the benchmark line and the reference arm, 10 for --hx-only, 3 for --warm, 2 for --batch, 1 for --big)")
    ap.add_argument("--warmup", type=int, default=None, help="untimed warm-up steps (default 3; 1 for --big)")
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--workload", default=WORKLOAD)
    ap.add_argument("--tol", type=float, default=1e-5,
                    help="|beta_1/alpha_1| stopping tolerance (the paper's default Lanc_Error)")
    ap.add_argument("--window", type=int, default=20)
    ap.add_argument("--e2e-steps", type=int, default=3)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-fp64", action="store_true", help="skip the plain-FP64 comparison solves")
    ap.add_argument("--states", action="store_true",
                    help="the three lowest states of the default workload (locking), mixed and FP64")
    ap.add_argument("--truncate", action="store_true",
                    help="truncated model space (Sec. 3.5): E0 and time at nested Dimension_Limit values")
    ap.add_argument("--hx-only", action="store_true",
                    help="time only the H*x kernel (profiling aid; not the benchmark line)")
    ap.add_argument("--omega", type=int, default=0, help="with --hx-only: picket-fence size instead of --workload")
    ap.add_argument("--npairs", type=int, default=0)
    ap.add_argument("--precision", choices=["fp32", "fp64"], default="fp32")
    ap.add_argument("--hx-variant", type=int, default=0, help="H*x kernel variant (0 = automatic)")
    ap.add_argument("--low-bits", type=int, default=0, help="orbits per basis block (0 = automatic)")
    ap.add_argument("--batch", action="store_true",
                    help="4096-problem mean-field workload: solves/s and per-solve latency (own JSON line)")
    ap.add_argument("--batch-count", type=int, default=4096)
    ap.add_argument("--big", action="store_true",
                    help="Omega=32, N=16 (dim 6.0e8): time-to-E0 of FP64, mixed and mixed+learned start")
    ap.add_argument("--odd", action="store_true",
                    help="odd-mass twin of the default workload (25 orbits, 12 pairs + 1 particle, Block = 0)")
    ap.add_argument("--warm", action="store_true",
                    help="Omega=30 workload: FP64 random start vs mixed + learned warm start (own JSON line)")
    ap.add_argument("--train-problems", type=int, default=240)
    ap.add_argument("--train-steps", type=int, default=2500)
    ap.add_argument("--no-mlp", action="store_true", help="batch mode without the learned warm start")
    ap.add_argument("--no-omega30", action="store_true",
                    help="default line without the Omega=30 forms (FP64 vs mixed vs mixed + learned start)")
    ap.add_argument("--omega30-steps", type=int, default=3)
    ap.add_argument("--no-autotune", action="store_true",
                    help="skip tuning the H*x schedule of the workload before the timed solves")
    return ap.parse_args()


# ----------------------------------------------------------------- helpers --
def combine_ranks(ms: float, nnz: float, dist, device: str = "cuda"):
    """Replicas: the slowest rank's time and the nonzeros of all ranks (every
    rank calls this; the whole-job throughput is their quotient)."""
    import torch
    t = torch.tensor([ms, nnz], dtype=torch.float64, device=device)
    tmax = t.clone()
    dist.all_reduce(tmax, op=dist.ReduceOp.MAX)
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(tmax[0]), float(t[1])


def dist_env():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return world, rank, local


def measured_peaks():
    f = ROOT / "MEASURED_PEAKS.json"
    if f.exists():
        d = json.loads(f.read_text())
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi sampling of SM clocks and throttle reasons during the timed region."""
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index: int):
        self.tmp = tempfile.NamedTemporaryFile("w+", suffix=".csv", delete=False)
        try:
            self.p = subprocess.Popen(["nvidia-smi", "-i", str(gpu_index), f"--query-gpu={self.FIELDS}",
                                       "--format=csv,noheader,nounits", "-lms", "200"],
                                      stdout=self.tmp, stderr=subprocess.DEVNULL)
        except FileNotFoundError:
            self.p = None

    def stop(self) -> dict:
        if self.p is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.p.terminate()
        try:
            self.p.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.p.kill()
        self.tmp.flush()
        rows = [r.split(",") for r in Path(self.tmp.name).read_text().splitlines() if r.strip()]
        os.unlink(self.tmp.name)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in rows:
            r = [c.strip() for c in r]
            try:
                sm.append(float(r[1]))
                smax.append(float(r[2]))
            except (ValueError, IndexError):
                continue
            for i, nm in enumerate(names):
                if len(r) > 5 + i and r[5 + i].lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "samples": len(sm), "reasons": sorted(reasons)}


def hx_roof(nnz: int, dim: int, es: int, seconds: float, fma_tflops: float, hbm_gbs: float) -> dict:
    """A product against its floor: one multiply-add per nonzero at the rate that
    the device reaches in that precision (or x and y moved once, if that is longer)."""
    fma_s, hbm_s = 2.0 * nnz / (fma_tflops * 1e12), 2.0 * dim * es / (hbm_gbs * 1e9)
    alu = fma_s >= hbm_s
    return {"bound": "fma" if alu else "hbm",
            "achieved": 2.0 * nnz / seconds / 1e12 if alu else 2.0 * dim * es / seconds / 1e9,
            "peak": fma_tflops if alu else hbm_gbs, "unit": "TFLOP/s" if alu else "GB/s",
            "frac": max(fma_s, hbm_s) / seconds, "fma_floor_ms": fma_s * 1e3, "hbm_floor_ms": hbm_s * 1e3,
            "avg_launch_ms": seconds * 1e3, "hx_nnz_per_s": nnz / seconds}


def hx_source_hash() -> str:
    h = hashlib.sha256()
    for f in ("pd_hx.cu", "pd_hxf.cu", "pd_internal.h"):
        h.update((ROOT / "paper_2001_01978_gb300" / "csrc" / f).read_bytes())
    return h.hexdigest()[:16]


def ncu_traffic(workload: str, precision: str, low_bits: int, variant: int):
    """DRAM bytes per H*x launch of this schedule from the committed ncu summary,
    or None when there is none or the kernel source changed since the capture."""
    f = ROOT / "profiles" / "hx_traffic.txt"
    if not f.exists():
        return None
    for line in f.read_text().splitlines():
        parts = line.split()
        if len(parts) >= 6 and not line.startswith("#") and parts[:4] == [workload, precision, str(low_bits), str(variant)]:
            return float(parts[4]) if parts[5] == hx_source_hash() else None
    return None


# ------------------------------------------------------------- CPU oracle ---
def oracle_hx_sample(omega, n, e, G, budget_s: float, seed: int = 0):
    """Time the oracle's H*x (binary-search scattering) on a bounded sample of
    contiguous rows; returns (nnz/s, rows, seconds, threads)."""
    import oracle
    b = oracle.basis(omega, n)
    dim = len(b)
    x = pd_inputs.random_vector(dim, 5)
    per_row = n * (omega - n)
    rows_n = min(dim, 20000)
    start = 0
    # grow the sample until it costs about budget_s
    while True:
        rows = np.arange(start, start + rows_n, dtype=np.int64)
        t0 = time.perf_counter()
        oracle.hx_rows(omega, n, e, G, x, rows, b)
        dt = time.perf_counter() - t0
        if dt >= 0.5 * budget_s or rows_n >= dim:
            break
        rows_n = min(dim, int(rows_n * max(2.0, 0.8 * budget_s / max(dt, 1e-3))))
    threads = int(os.environ.get("OMP_NUM_THREADS", os.cpu_count() or 1))
    return rows_n * per_row / dt, rows_n, dt, threads


def run_reference(args):
    world, rank, _ = dist_env()
    if rank != 0:
        return 0
    omega, n, e, G = pd_inputs.workload(args.workload)
    import oracle
    b = oracle.basis(omega, n)
    dim = len(b)
    x = pd_inputs.random_vector(dim, 5)
    per_row = n * (omega - n)
    # one step = the oracle's H*x over a fixed block of rows sized to ~2 s
    rows_n = min(dim, 20000)
    while True:
        rows = np.arange(0, rows_n, dtype=np.int64)
        t0 = time.perf_counter()
        oracle.hx_rows(omega, n, e, G, x, rows, b)
        dt = time.perf_counter() - t0
        if dt >= 1.0 or rows_n >= dim:
            break
        rows_n = min(dim, int(rows_n * max(2.0, 1.5 / max(dt, 1e-3))))
    rng = np.random.default_rng(0)
    offsets = [int(v) for v in rng.integers(0, max(1, dim - rows_n), size=args.warmup + args.steps)]
    for i in range(args.warmup):
        oracle.hx_rows(omega, n, e, G, x, np.arange(offsets[i], offsets[i] + rows_n, dtype=np.int64), b)
    t0 = time.perf_counter()
    for i in range(args.steps):
        o = offsets[args.warmup + i]
        oracle.hx_rows(omega, n, e, G, x, np.arange(o, o + rows_n, dtype=np.int64), b)
    dt = time.perf_counter() - t0
    value = args.steps * rows_n * per_row / dt
    threads = int(os.environ.get("OMP_NUM_THREADS", os.cpu_count() or 1))
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * dt / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": args.workload, "omega": omega, "n_pairs": n, "dim": dim,
                   "rows_per_step": rows_n, "l2": "CPU run"},
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": threads, "kind": "oracle",
                         "sample": f"oracle H*x (binary-search scattering) over {rows_n} contiguous rows per step"},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))
    return 0


# -------------------------------------------------------------- GPU path ----
def run_ours(args):
    import torch
    world, rank, local = dist_env()
    torch.cuda.set_device(local)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    def barrier():
        if dist is not None:
            dist.barrier()

    import paper_2001_01978_gb300 as pd

    omega, n, e, G = pd_inputs.workload(args.workload)
    dim = math.comb(omega, n)
    nnz = dim * n * (omega - n)
    stream = torch.cuda.current_stream()
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")

    def make(prec):
        s = pd.Solver(omega, n, e, G, precision=prec, window=args.window, start=pd.PD_START_RANDOM, seed=1,
                      hx_variant=args.hx_variant, low_bits=args.low_bits)
        pd.pairdiag_set_stream(s.h, stream)
        return s

    tuned = None
    if not args.no_autotune:
        tuned = {}
        for pname, prec in (("fp32", pd.PD_PREC_MIXED), ("fp64", pd.PD_PREC_FP64)):
            best, cands = pd.pairdiag_autotune(omega, n, e, G, prec, reps=5)
            tuned[pname] = {"best": best, "candidates": cands}
    # the chosen form: mixed precision from the learned warm start (trained once,
    # outside the timed region, on ground states the solver computes at Omega <= 18)
    ws, train_s, l0, l1, trows = (None, None, None, None, None) if args.no_mlp else train_warm_start(args.train_problems, args.train_steps)
    mixed = make(pd.PD_PREC_MIXED)
    if ws is not None:
        mixed.close()
        mixed = pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, window=args.window,
                          start=pd.PD_START_MLP, seed=1, hx_variant=args.hx_variant, low_bits=args.low_bits)
        pd.pairdiag_set_stream(mixed.h, stream)
        ws.attach(mixed.h)
    mixed_rand = None if ws is None else make(pd.PD_PREC_MIXED)
    fp64 = None if args.no_fp64 else make(pd.PD_PREC_FP64)

    def solve(s):
        return pd.pairdiag_ground_state_dev(s.h, args.tol, None)

    for _ in range(args.warmup):
        flush.fill_(1.0)
        r = solve(mixed)
        if mixed_rand is not None:
            solve(mixed_rand)
        if fp64 is not None:
            solve(fp64)

    # ---- timed region: K mixed solves ----
    pd.pairdiag_set_profiling(mixed.h, True)
    pd.pairdiag_get_profile(mixed.h, -1)      # clear
    clocks = ClockSampler(local)
    launches0 = pd.pairdiag_kernel_launches()
    barrier()
    torch.cuda.synchronize()
    wall0 = time.perf_counter()
    step_ms, results = [], []
    for _ in range(args.steps):
        flush.fill_(1.0)
        ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        ev0.record(stream)
        r = solve(mixed)
        ev1.record(stream)
        ev1.synchronize()
        step_ms.append(ev0.elapsed_time(ev1))
        results.append(r)
    torch.cuda.synchronize()
    barrier()
    wall = time.perf_counter() - wall0
    launches = pd.pairdiag_kernel_launches() - launches0
    clk = clocks.stop()
    hx_count, hx_ms = pd.pairdiag_get_profile(mixed.h)
    hx64_count, hx64_ms = pd.pairdiag_get_profile(mixed.h, pd.PD_PREC_FP64)   # the FP64 refinement products
    # the vector work of the Lanczos steps that follow the products
    st32_count, st32_ms = pd.pairdiag_get_profile(mixed.h, pd.PD_PROF_STEP + pd.PD_PREC_MIXED)
    st64_count, st64_ms = pd.pairdiag_get_profile(mixed.h, pd.PD_PROF_STEP + pd.PD_PREC_FP64)
    pd.pairdiag_set_profiling(mixed.h, False)

    total_ms = sum(step_ms)
    products = sum(r["hx_products"] for r in results)
    nnz_done = products * nnz
    if dist is not None:
        total_ms_max, nnz_all = combine_ranks(total_ms, float(nnz_done), dist, "cuda")
    else:
        total_ms_max, nnz_all = total_ms, float(nnz_done)
    value = nnz_all / (total_ms_max * 1e-3)

    def timed(s):
        ms, res = [], []
        for _ in range(args.steps):
            flush.fill_(1.0)
            ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            ev0.record(stream)
            r = solve(s)
            ev1.record(stream)
            ev1.synchronize()
            ms.append(ev0.elapsed_time(ev1))
            res.append(r)
        return ms, res

    # ---- comparison forms: mixed from a random start, plain FP64 Lanczos ----
    mr_ms, mr_res = timed(mixed_rand) if mixed_rand is not None else ([], [])
    fp64_ms, fp64_res = timed(fp64) if fp64 is not None else ([], [])

    # ---- end to end through the public API with host buffers ----
    e2e_s, e2e_hx = [], []
    Bi = (omega + omega * omega) * 8
    Bo = dim * 8 + 8
    vec_host = torch.empty(dim, dtype=torch.float64, pin_memory=True).numpy()   # the caller's output buffer
    barrier()                                  # replicas start their end-to-end solves together
    for _ in range(max(1, args.e2e_steps)):
        flush.fill_(1.0)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, window=args.window, seed=1,
                       start=pd.PD_START_MLP if ws is not None else pd.PD_START_RANDOM,
                       hx_variant=args.hx_variant, low_bits=args.low_bits) as s:
            if ws is not None:
                ws.attach(s.h)
            r = s.ground_state(args.tol, want_vector=True, out=vec_host)   # E0 + eigenvector into pinned host memory
        e2e_s.append(time.perf_counter() - t0)
        e2e_hx.append(r["hx_products"])
    if dist is not None:
        # whole job: the nonzeros of every replica over the slowest replica's time
        e2e_ms_max, e2e_nnz_all = combine_ranks(1e3 * sum(e2e_s), float(sum(e2e_hx) * nnz), dist, "cuda")
        e2e_value = e2e_nnz_all / (e2e_ms_max * 1e-3)
    else:
        e2e_value = sum(e2e_hx) * nnz / sum(e2e_s)

    # ---- the Omega=30 workload (dim 1.55e8) in the three forms: FP64 from a random
    # start, mixed from a random start, mixed from the learned start ----
    om30 = None
    if not args.no_omega30 and ws is not None:
        om30 = forms_on(args, "omega30_n15_sepnoise_s2", ws, args.omega30_steps, 1, kato_temple=True)
    # ---- ALU roof of the FP64 product (one FP64 FMA per nonzero) ----
    fma64 = pd.pairdiag_fma_peak(pd.PD_PREC_FP64, 5, stream)

    def close_all():
        for s_ in (mixed, mixed_rand, fp64):
            if s_ is not None:
                s_.close()
        if ws is not None:
            ws.close()
        if dist is not None:
            dist.destroy_process_group()

    if rank != 0:
        close_all()
        return 0

    # ---- accuracy against the oracle's E0 (committed by tests/golden/make_golden.py) ----
    e0 = results[-1]["e0"]
    golden = ROOT / "tests" / "golden" / f"{args.workload}_e0.txt"
    rel_err = None
    if golden.exists():
        vals = [l.split() for l in golden.read_text().splitlines() if l.strip() and not l.startswith("#")]
        e_ref = float(vals[0][0])
        rel_err = abs(e0 - e_ref) / abs(e_ref)

    # ---- roofline of the dominant kernel (FP32 H*x) ----
    peak, peak_kind = measured_peaks()
    fma32 = pd.pairdiag_fma_peak(pd.PD_PREC_MIXED, 5, stream)
    # per executed FP32 product: launches skipped after a cycle ended early (a
    # converged Ritz pair) add their few microseconds to hx_ms, not to the count
    hx_executed = sum(r["iterations_fp32"] for r in results)
    avg_hx_s = (hx_ms / max(1, hx_executed)) * 1e-3
    lb, hv = pd.pairdiag_tune_get(omega, n, pd.PD_PREC_MIXED)
    if args.low_bits or args.hx_variant:
        lb, hv = args.low_bits, args.hx_variant
    # a zero (no recorded or requested value, e.g. --no-autotune) is left to the
    # library's untuned default, which no traffic line describes
    traffic = ncu_traffic(args.workload, "fp32", lb, hv) if lb and hv else None
    kname = "H*x FP32 (low_bits %s, variant %s)" % (lb or "default", hv or "default")
    # The floor of a product: one multiply-add per nonzero at the measured FP32 rate
    # (x read and y written once take a tenth of that, hbm_floor_ms).  traffic: the
    # DRAM bytes ncu counts per product.
    roofline = dict(hx_roof(nnz, dim, 4, avg_hx_s, fma32, peak),
                **{"kernel": kname, "peak_kind": "measured (pairdiag_fma_peak)", "hbm_peak_gbs": peak,
                "hbm_peak_kind": peak_kind, "traffic": traffic, "dram_gbs": (traffic / avg_hx_s / 1e9) if traffic else None,
                "hx_share_of_step": (hx_ms + hx64_ms) / total_ms,
                "hx32_share_of_step": hx_ms / total_ms,
                "hx_share_is": "all H*x products of a solve (FP32 cycles + FP64 refinement) / solve time",
                "timed_launches": hx_count, "executed_products": hx_executed,
                "step_share_of_step": (st32_ms + st64_ms) / total_ms,
                "step_avg_ms": (st32_ms + st64_ms) / max(1, st32_count + st64_count),
                "step_share_is": "vector work of the Lanczos steps after each product (recurrence, "
                                 "full Gram-Schmidt pass, norm, next basis vector) / solve time"})

    cpu = None
    if not args.no_cpu_baseline and world == 1:
        v, rows_n, dt, threads = oracle_hx_sample(omega, n, e, G, budget_s=12.0)
        cpu = {"value": v, "unit": UNIT, "cores": threads, "kind": "oracle",
               "sample": f"oracle H*x (binary-search scattering) over {rows_n} contiguous rows, {dt:.1f} s"}

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32+f64", "data": "synthetic",
        "config": {"workload": args.workload, "omega": omega, "n_pairs": n, "dim": dim,
                   "nnz_offdiag_per_hx": nnz,
                   "form": "mixed" + ("+learned warm start" if ws is not None else ""), "tol": args.tol,
                   "window": args.window,
                   "start": "learned warm start" if ws is not None else "random (SplitMix64, seed 1)",
                   "l2": "flushed between steps (512 MB write)",
                   "parallelism": "replicas" if world > 1 else "single"},
        "autotune": tuned,
        "warm_start_training": None if ws is None else {"problems": args.train_problems, "rows": trows,
                                                         "seconds": train_s, "loss_first": l0, "loss_last": l1},
        "e0": e0, "e0_fp64": fp64_res[-1]["e0"] if fp64_res else None,
        "hx_per_step": products / args.steps,
        "iterations": {"chosen": results[-1]["iterations"], "chosen_fp32": results[-1]["iterations_fp32"],
                       "mixed_random_start": mr_res[-1]["iterations"] if mr_res else None,
                       "fp64_random_start": fp64_res[-1]["iterations"] if fp64_res else None},
        "wall_s_timed_region": wall,
        "omega30_detail": om30,
        "fp64_hx_alu_roof": {"fma_peak_tflops": fma64,
                             "omega30_fp64_hx_frac": (om30["roof"]["fp64"]["hx_nnz_per_s"] * 2e-12 / fma64)
                             if om30 and "fp64" in om30["roof"] else None},
    }
    if om30 is not None:
        f30 = om30["forms"]
        line["omega30"] = {
            "ms": {k: round(v["time_to_e0_ms"], 1) for k, v in f30.items()},
            "iters": {k: v["iterations"] for k, v in f30.items()},
            "speedup_mixed_mlp_vs_fp64": f30["fp64_random"]["time_to_e0_ms"] / f30["mixed_mlp"]["time_to_e0_ms"],
            "kato_temple_rel": {k: v["kato_temple_rel_bound"] for k, v in f30.items()},
            "hx_frac": {k: round(v["frac"], 3) for k, v in om30["roof"].items()}}
    line.update({
        "time_to_e0_ms": {"chosen": statistics.mean(step_ms),
                          "mixed_random_start": statistics.mean(mr_ms) if mr_ms else None,
                          "fp64_random_start": statistics.mean(fp64_ms) if fp64_ms else None},
        "speedup_chosen_vs_fp64": (statistics.mean(fp64_ms) / statistics.mean(step_ms)) if fp64_ms else None,
        "e0_rel_err_vs_oracle": rel_err,
        "roofline": roofline,
        "cpu_baseline": cpu,
        "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": Bi, "d2h_bytes_per_step": Bo,
                "ms_per_step": 1e3 * statistics.mean(e2e_s),
                "what": "pairdiag_create + pairdiag_ground_state (E0 and eigenvector to pinned host memory) + destroy"},
        "gpu_launches": launches,
        "clocks": clk,
    })
    print(json.dumps(line))
    close_all()
    return 0


def run_hx_only(args):
    """K back-to-back H*x launches on resident vectors, each timed with CUDA events."""
    import torch
    import paper_2001_01978_gb300 as pd
    torch.cuda.set_device(0)
    if args.omega:
        omega, n = args.omega, args.npairs
        e, G = pd_inputs.separable_noise(omega, seed=1)
        name = f"omega{omega}_n{n}_sepnoise_s1"
    else:
        omega, n, e, G = pd_inputs.workload(args.workload)
        name = args.workload
    dim = math.comb(omega, n)
    nnz = dim * n * (omega - n)
    prec = pd.PD_PREC_MIXED if args.precision == "fp32" else pd.PD_PREC_FP64
    dt = torch.float32 if prec == pd.PD_PREC_MIXED else torch.float64
    es = 4 if prec == pd.PD_PREC_MIXED else 8
    with pd.Solver(omega, n, e, G, hx_variant=args.hx_variant, low_bits=args.low_bits) as s:
        stream = torch.cuda.current_stream()
        pd.pairdiag_set_stream(s.h, stream)
        g = torch.Generator(device="cuda").manual_seed(1)
        x = torch.randn(dim, dtype=dt, device="cuda", generator=g)
        y = torch.empty_like(x)
        flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
        for _ in range(args.warmup):
            pd.pairdiag_hx_dev(s.h, prec, x, y)
        times = []
        for _ in range(args.steps):
            flush.fill_(1.0)
            ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            ev0.record(stream)
            pd.pairdiag_hx_dev(s.h, prec, x, y)
            ev1.record(stream)
            ev1.synchronize()
            times.append(ev0.elapsed_time(ev1))
    ms = statistics.median(times)
    peak, kind = measured_peaks()
    roof = hx_roof(nnz, dim, es, ms * 1e-3, pd.pairdiag_fma_peak(prec, 5, stream), peak)
    print(json.dumps({"hx_only": True, "workload": name, "precision": args.precision, "dim": dim,
                      "hx_variant": args.hx_variant, "low_bits": args.low_bits,
                      "nnz": nnz, "median_ms": ms, "min_ms": min(times), "nnz_per_s": nnz / (ms * 1e-3),
                      "roofline": roof, "hbm_peak_kind": kind,
                      "l2": "flushed before each launch"}))
    return 0


def train_warm_start(count: int, steps: int = 2500):
    """One-off: train the warm-start network on ground states the solver computes
    at Omega <= 18 (returns the network and the seconds it took)."""
    from paper_2001_01978_gb300 import warmstart
    t0 = time.perf_counter()
    X, T = warmstart.training_set(pd_inputs.training_problems(count, seed=11, omega_lo=10, omega_hi=18))
    ws = warmstart.WarmStart(seed=0)
    hist = ws.train(X, T, steps=steps, lr=2e-3)
    return ws, time.perf_counter() - t0, float(hist[0]), float(hist[-1]), len(X)


def run_warm(args):
    """Omega=30, N=15 (dim 1.55e8, seed 2): time-to-E0 and Lanczos iterations of
    plain FP64 Lanczos from a random start vs the mixed form from the learned
    warm start (and from a random start), same tolerance."""
    return run_forms(args, "omega30_n15_sepnoise_s2", "warm_start")


def run_big(args):
    """Omega=32, N=16 (dim 6.0e8, seed 3), the largest single solve: the same
    three forms, each on its own (their windows do not fit on the device
    together), with the in-situ H*x roofline of both precisions."""
    return run_forms(args, "omega32_n16_constnoise_s3", "largest_single_solve")


def forms_on(args, workload, ws, steps, warmup, kato_temple=False):
    """Time-to-E0 of three forms on one workload: plain FP64 from a random start,
    mixed from a random start, mixed from the learned warm start.  One solver per
    form, created, warmed up (first touch of the window and FP64 vectors), timed
    over `steps` solves and closed before the next form.  With kato_temple, the
    FP64 Rayleigh quotient of each returned vector and its residual r give the
    Kato-Temple bound r^2/gap of its E0 error (the library's FP64 H*x, which the
    GPU tests pin row by row against the oracle at this size; gap from the
    second Ritz value)."""
    import torch
    import paper_2001_01978_gb300 as pd
    omega, n, e, G = pd_inputs.workload(workload)
    dim = math.comb(omega, n)
    nnz = dim * n * (omega - n)
    stream = torch.cuda.current_stream()
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
    tuned = {}
    if not args.no_autotune:
        for pname, prec in (("fp32", pd.PD_PREC_MIXED), ("fp64", pd.PD_PREC_FP64)):
            best, _ = pd.pairdiag_autotune(omega, n, e, G, prec, reps=3)
            tuned[pname] = best
    forms = [("fp64_random", pd.PD_PREC_FP64, pd.PD_START_RANDOM),
             ("mixed_random", pd.PD_PREC_MIXED, pd.PD_START_RANDOM),
             ("mixed_mlp", pd.PD_PREC_MIXED, pd.PD_START_MLP)]
    peak, _ = measured_peaks()
    out, roof = {}, {}
    for name, prec, start in forms:
        with pd.Solver(omega, n, e, G, precision=prec, start=start, window=args.window, seed=1) as s:
            pd.pairdiag_set_stream(s.h, stream)
            if start == pd.PD_START_MLP:
                ws.attach(s.h)
            for _ in range(warmup):
                flush.fill_(1.0)
                pd.pairdiag_ground_state_dev(s.h, args.tol, None)
            pd.pairdiag_set_profiling(s.h, True)
            pd.pairdiag_get_profile(s.h, -1)              # clear
            times, r, executed = [], None, 0
            v = torch.empty(dim, dtype=torch.float64, device="cuda") if kato_temple else None
            for i in range(max(1, steps)):
                flush.fill_(1.0)
                ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                ev0.record(stream)
                r = pd.pairdiag_ground_state_dev(s.h, args.tol, v)
                ev1.record(stream)
                ev1.synchronize()
                times.append(ev0.elapsed_time(ev1))
                # products of the profiled precision that ran (not skipped launches)
                executed += r["hx_products"] if prec == pd.PD_PREC_FP64 else r["iterations_fp32"]
            pkey = "fp64" if prec == pd.PD_PREC_FP64 else "fp32"
            cnt, ms = pd.pairdiag_get_profile(s.h, pd.PD_PREC_FP64 if pkey == "fp64" else pd.PD_PREC_MIXED)
            pd.pairdiag_set_profiling(s.h, False)
            kt = None
            if kato_temple:
                w = torch.empty_like(v)
                pd.pairdiag_hx_dev(s.h, pd.PD_PREC_FP64, v, w)
                lam = float(v @ w) / float(v @ v)
                res = float(torch.linalg.vector_norm(w - lam * v)) / float(torch.linalg.vector_norm(v))
                kt = res * res / max(r["gap_estimate"], 1e-12) / abs(lam)
                del w
            del v
            if cnt and pkey not in roof:
                avg_s = ms / max(1, executed) * 1e-3
                fma = pd.pairdiag_fma_peak(pd.PD_PREC_FP64 if pkey == "fp64" else pd.PD_PREC_MIXED, 5, stream)
                roof[pkey] = dict(hx_roof(nnz, dim, 8 if pkey == "fp64" else 4, avg_s, fma, peak),
                                  timed_launches=cnt, executed_products=executed)
        out[name] = {"time_to_e0_ms": statistics.median(times), "iterations": r["iterations"],
                     "iterations_fp32": r["iterations_fp32"], "hx_products": r["hx_products"],
                     "nnz_per_s": r["hx_products"] * nnz / (statistics.median(times) * 1e-3),
                     "e0": r["e0"], "rel_residual": r["rel_residual"], "status": r["status"],
                     "kato_temple_rel_bound": kt}
    ref = out["fp64_random"]["e0"]
    for v_ in out.values():
        v_["e0_rel_diff_vs_fp64"] = abs(v_["e0"] - ref) / abs(ref)
    return dict(workload=workload, omega=omega, n_pairs=n, dim=dim, nnz=nnz, tuned=tuned, forms=out, roof=roof)


def run_forms(args, workload, tag):
    """The three forms of forms_on, each timed over --steps solves after --warmup."""
    import torch
    torch.cuda.set_device(0)
    ws, train_s, l0, l1, rows = train_warm_start(args.train_problems, args.train_steps)
    clocks = ClockSampler(0)
    f = forms_on(args, workload, ws, args.steps, args.warmup, kato_temple=True)
    clk = clocks.stop()
    out = f["forms"]
    print(json.dumps({tag: True, "workload": workload, "omega": f["omega"], "n_pairs": f["n_pairs"], "dim": f["dim"],
                      "nnz_offdiag_per_hx": f["nnz"], "tol": args.tol, "window": args.window,
                      "steps": args.steps, "warmup": args.warmup,
                      "l2": "flushed between solves (512 MB write)",
                      "training": {"problems": args.train_problems, "rows": rows, "seconds": train_s,
                                   "loss_first": l0, "loss_last": l1},
                      "autotune": f["tuned"], "forms": out, "hx_roofline": f["roof"], "clocks": clk,
                      "speedup_mixed_mlp_vs_fp64_random": out["fp64_random"]["time_to_e0_ms"] / out["mixed_mlp"]["time_to_e0_ms"]}))
    ws.close()
    return 0


def run_truncate(args):
    """The truncated model space of Sec. 3.5 on the Omega=28, N=14 separable
    workload (seed 1, dim 4.0e7): for nested Dimension_Limit values, the kept
    dimension, the set-up time of the truncation (diagonal histogram and kept
    map), the time of one truncated FP32 H*x, the time to E0 of the mixed form
    and E0 against the full-space E0 (the convergence Sec. 5.4 studies)."""
    import torch
    import paper_2001_01978_gb300 as pd
    torch.cuda.set_device(0)
    omega, n = 28, 14
    e, G = pd_inputs.separable_noise(omega, seed=1)
    dim = math.comb(omega, n)
    stream = torch.cuda.current_stream()
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
    rows = []
    clocks = ClockSampler(0)
    with pd.Solver(omega, n, e, G, precision=pd.PD_PREC_MIXED, window=args.window, seed=1) as s:
        pd.pairdiag_set_stream(s.h, stream)
        full = pd.pairdiag_ground_state_dev(s.h, 1e-9, None)
        for limit in (10 ** 5, 10 ** 6, 4 * 10 ** 6, 10 ** 7, 0):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            kept = pd.pairdiag_truncate(s.h, limit)
            t_setup = time.perf_counter() - t0
            x = torch.randn(kept, dtype=torch.float32, device="cuda")
            y = torch.empty_like(x)
            for _ in range(2):
                pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, x, y)
            hx_ms = []
            for _ in range(3):
                flush.fill_(1.0)
                ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                ev0.record(stream)
                pd.pairdiag_hx_dev(s.h, pd.PD_PREC_MIXED, x, y)
                ev1.record(stream)
                ev1.synchronize()
                hx_ms.append(ev0.elapsed_time(ev1))
            del x, y
            flush.fill_(1.0)
            ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            ev0.record(stream)
            r = pd.pairdiag_ground_state_dev(s.h, 1e-9, None)
            ev1.record(stream)
            ev1.synchronize()
            rows.append({"dimension_limit": limit or None, "kept_dim": kept, "nnz": pd.pairdiag_nnz(s.h),
                         "setup_s": t_setup, "hx_ms": statistics.median(hx_ms),
                         "hx_nnz_per_s": pd.pairdiag_nnz(s.h) / (statistics.median(hx_ms) * 1e-3),
                         "time_to_e0_ms": ev0.elapsed_time(ev1), "iterations": r["iterations"], "e0": r["e0"],
                         "e0_minus_full": r["e0"] - full["e0"], "status": r["status"]})
    clk = clocks.stop()
    print(json.dumps({"truncation": True, "workload": "omega28_n14_sepnoise_s1", "dim": dim, "tol": 1e-9,
                      "form": "mixed", "bins": 10 ** 8, "full_e0": full["e0"], "limits": rows, "clocks": clk}))
    return 0


def run_batch(args):
    """Batched form: 4096 Hamiltonians (Omega ~ U{10..22}, N = Omega/2 +- U{0..3}) in
    one lock-step solve, mixed form vs plain FP64, same tolerance."""
    import torch
    import paper_2001_01978_gb300 as pd
    torch.cuda.set_device(0)
    probs = pd_inputs.batch_workload(args.batch_count, seed=5)
    dims = [math.comb(om, n) for om, n, _, _ in probs]
    nnz = sum(d * n * (om - n) for d, (om, n, _, _) in zip(dims, probs))
    stream = torch.cuda.current_stream()
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
    ws, train_s = (None, None) if args.no_mlp else train_warm_start(args.train_problems, args.train_steps)[:2]
    forms = [("mixed", pd.PD_PREC_MIXED, pd.PD_START_RANDOM), ("fp64", pd.PD_PREC_FP64, pd.PD_START_RANDOM)]
    if ws is not None:
        forms.insert(0, ("mixed_mlp", pd.PD_PREC_MIXED, pd.PD_START_MLP))
    # the oracle's E0 of twelve stratified problems (tests/golden/make_golden.py)
    picks_ref = {}
    gf = ROOT / "tests" / "golden" / f"batch{len(probs)}_s5_picks_e0.txt"
    if gf.exists():
        for line in gf.read_text().splitlines():
            if line.strip() and not line.startswith("#"):
                row = line.split()
                picks_ref[int(row[0])] = float(row[4])
    out = {}
    for name, prec, start in forms:
        opt = pd.pairdiag_default_options(precision=prec, window=args.window, start=start,
                                          hx_variant=args.hx_variant)
        mlp = ws.m if start == pd.PD_START_MLP else None
        for _ in range(max(1, args.warmup // 3)):
            pd.pairdiag_batch_ground_state(probs, args.tol, opt, stream, mlp)
        times, res = [], None
        for _ in range(args.steps):
            flush.fill_(1.0)
            ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            ev0.record(stream)
            res = pd.pairdiag_batch_ground_state(probs, args.tol, opt, stream, mlp)
            ev1.record(stream)
            ev1.synchronize()
            times.append(ev0.elapsed_time(ev1))
        ms = statistics.median(times)
        lat = res["latency_ms"]
        iters = res["iterations"]
        errs = [abs(res["e0"][i] - ref) / abs(ref) for i, ref in picks_ref.items()]
        out[name] = {"batch_ms": ms, "solves_per_s": len(probs) / (ms * 1e-3),
                     "latency_ms_p50": float(np.percentile(lat, 50)), "latency_ms_p99": float(np.percentile(lat, 99)),
                     "converged_frac": float(np.mean(res["converged"])),
                     "iterations_mean": float(np.mean(iters)), "iterations_max": int(np.max(iters)),
                     "e0_max_rel_err_vs_oracle": max(errs) if errs else None,
                     "oracle_picks": len(errs)}
    e_m = np.array([0.0])
    print(json.dumps({"batch": True, "workload": "mean-field batch: %d problems, Omega ~ U{10..22}, seed 5" % len(probs),
                      "total_dim": int(sum(dims)), "nnz_offdiag_per_batched_hx": int(nnz), "tol": args.tol,
                      "window": args.window, "steps": args.steps, "l2": "flushed between steps",
                      "warm_start_training_s": train_s,
                      "mixed_mlp": out.get("mixed_mlp"), "mixed": out["mixed"], "fp64": out["fp64"],
                      "speedup_mixed_vs_fp64": out["fp64"]["batch_ms"] / out["mixed"]["batch_ms"],
                      "speedup_mixed_mlp_vs_fp64": (out["fp64"]["batch_ms"] / out["mixed_mlp"]["batch_ms"]
                                                    if "mixed_mlp" in out else None)}))
    if ws is not None:
        ws.close()
    return 0


def run_odd(args):
    """Odd-mass twin of the default workload: 25 orbits (separable G plus noise, seed
    1), 12 pairs and one unpaired particle, every blocked subspace solved (the
    paper's Block = 0, Eq. 3): 25 subspaces of C(24,12) = 2.7e6 states each.
    Time to the lowest E_b: plain FP64, the mixed form, and the mixed form from
    the learned warm start (the network trained once, outside the timing), same
    tolerance."""
    import torch
    import paper_2001_01978_gb300 as pd
    torch.cuda.set_device(0)
    ws = None if args.no_mlp else train_warm_start(args.train_problems, args.train_steps)[0]
    omega, n = 25, 12
    e, G = pd_inputs.separable_noise(omega, seed=1)
    dim = math.comb(omega - 1, n)
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
    out = {}
    clocks = ClockSampler(0)
    forms = [("mixed", pd.PD_PREC_MIXED, pd.PD_START_RANDOM), ("fp64", pd.PD_PREC_FP64, pd.PD_START_RANDOM)]
    if ws is not None:
        forms.insert(0, ("mixed_mlp", pd.PD_PREC_MIXED, pd.PD_START_MLP))
    for name, prec, start in forms:
        opt = pd.pairdiag_default_options(precision=prec, window=args.window, seed=1, start=start)
        mlp = ws.m if start == pd.PD_START_MLP else None
        for _ in range(args.warmup):
            pd.pairdiag_odd_ground_state(omega, n, e, G, args.tol, opt=opt, mlp=mlp, want_vector=False)
        times, r = [], None
        for _ in range(args.steps):
            flush.fill_(1.0)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            r = pd.pairdiag_odd_ground_state(omega, n, e, G, args.tol, opt=opt, mlp=mlp, want_vector=False)
            times.append((time.perf_counter() - t0) * 1e3)
        ms = statistics.median(times)
        out[name] = {"time_to_e0_ms": ms, "ms_per_subspace": ms / omega, "e0": r["e0"], "block": r["block"],
                     "winner_iterations": r["iterations"], "winner_rel_residual": r["rel_residual"],
                     "status": r["status"], "energies": [float(x) for x in r["energies"]]}
    clk = clocks.stop()
    for k in out:
        out[k]["e0_rel_diff_vs_fp64"] = abs(out[k]["e0"] - out["fp64"]["e0"]) / abs(out["fp64"]["e0"])
    # the oracle's E_b of one subspace (committed by tests/golden/make_golden.py)
    oracle_b = {}
    for f in sorted((ROOT / "tests" / "golden").glob(f"omega{omega}_n{n}_sepnoise_s1_odd_b*_e0.txt")):
        vals = [l.split() for l in f.read_text().splitlines() if l.strip() and not l.startswith("#")]
        oracle_b[int(f.name.split("_odd_b")[1].split("_")[0])] = float(vals[0][0])
    # every subspace with an oracle value, whichever block wins
    for v in out.values():
        v["e_b_rel_err_vs_oracle"] = {str(b): abs(v["energies"][b] - eb) / abs(eb) for b, eb in oracle_b.items()}
        del v["energies"]
    print(json.dumps({"odd_mass": True, "workload": "25 orbits, 12 pairs + 1 particle, separable G + noise, seed 1",
                      "subspaces": omega, "dim_per_subspace": dim, "tol": args.tol, "window": args.window,
                      "steps": args.steps, "warmup": args.warmup, "timing": "host wall clock around the "
                      "synchronous call (three host threads solve the subspaces, each on its own stream)",
                      "l2": "flushed between calls", "forms": out, "clocks": clk,
                      "speedup_mixed_vs_fp64": out["fp64"]["time_to_e0_ms"] / out["mixed"]["time_to_e0_ms"],
                      "speedup_mixed_mlp_vs_fp64": (out["fp64"]["time_to_e0_ms"] / out["mixed_mlp"]["time_to_e0_ms"]
                                                    if "mixed_mlp" in out else None)}))
    if ws is not None:
        ws.close()
    return 0


def run_states(args):
    """The lowest few states (Sec. 3.4, locking) of the default Omega=24 workload:
    time to the three lowest eigenpairs in the mixed form and in FP64 (tol 1e-8),
    the energies, and the orthonormality of the returned vectors."""
    import torch
    import paper_2001_01978_gb300 as pd
    torch.cuda.set_device(0)
    omega, n, e, G = pd_inputs.workload(args.workload)
    dim = math.comb(omega, n)
    k = 3
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
    stream = torch.cuda.current_stream()
    out = {}
    clocks = ClockSampler(0)
    for name, prec in (("mixed", pd.PD_PREC_MIXED), ("fp64", pd.PD_PREC_FP64)):
        with pd.Solver(omega, n, e, G, precision=prec, window=args.window, seed=1) as s:
            pd.pairdiag_set_stream(s.h, stream)
            vecs = torch.empty(k * dim, dtype=torch.float64, device="cuda")
            for _ in range(args.warmup):
                pd.pairdiag_lowest_states_dev(s.h, k, 1e-8, vecs)
            times, r = [], None
            for _ in range(args.steps):
                flush.fill_(1.0)
                ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                ev0.record(stream)
                r = pd.pairdiag_lowest_states_dev(s.h, k, 1e-8, vecs)
                ev1.record(stream)
                ev1.synchronize()
                times.append(ev0.elapsed_time(ev1))
            V = vecs.view(k, dim)
            gram = (V @ V.T).cpu().numpy()
        out[name] = {"ms": statistics.median(times), "energies": [float(x) for x in r["energies"]],
                     "iterations": [i["iterations"] for i in r["info"]], "status": r["status"],
                     "max_offdiag_overlap": float(np.max(np.abs(gram - np.eye(k))))}
    clk = clocks.stop()
    print(json.dumps({"lowest_states": True, "workload": args.workload, "dim": dim, "k": k, "tol": 1e-8,
                      "window": args.window, "steps": args.steps, "l2": "flushed between calls", "forms": out,
                      "clocks": clk}))
    return 0


def main():
    args = parse_args()
    mode = ("batch" if args.batch else "warm" if args.warm else "big" if args.big else "odd" if args.odd else
            "truncate" if args.truncate else "states" if args.states else
            "hx" if args.hx_only and args.impl != "reference" else "line")
    if args.steps is None:
        args.steps = {"batch": 2, "warm": 3, "big": 1, "hx": 10, "odd": 3, "states": 3, "truncate": 1}.get(mode, 30)
    if args.warmup is None:
        args.warmup = 1 if mode in ("big", "odd", "states", "truncate") else 3
    if args.batch:
        return run_batch(args)
    if args.warm:
        return run_warm(args)
    if args.big:
        return run_big(args)
    if args.odd:
        return run_odd(args)
    if args.truncate:
        return run_truncate(args)
    if args.states:
        return run_states(args)
    if args.impl == "reference":
        return run_reference(args)
    if args.hx_only:
        return run_hx_only(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
