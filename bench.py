#!/usr/bin/env python
"""Benchmark of the GB300 sparse Fast Chebyshev Transform hot path.

Headline workload (the metric's "mixed vs FP64" configuration): D=10,
total-degree-8 support (N = 43758 coefficients), rational target
1/(1 + sum c_i x_i^2) with seeded c_i ~ U[0.1, 1], on an L-grid of
L = 3D = 30 Chebyshev-extrema tensor grids drawn by Algorithm 1 (sizes in
{1..9}).  One step = one transform: per-grid DCT-I, bin gather, CGLS solve,
coefficients out, with the samples resident on the device before the timed
region and L2 flushed between steps.  Both paths run on the same samples: FP64
CG, and FP32 inner solves between FP64 refinement sweeps (mixed); `value` is
the faster path whose coefficients are within 1e-10 (relative l2) of the CPU
oracle's.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl gpu|reference]

Prints one JSON line (rank 0).  Under torchrun every rank solves its own
stream of transforms (replicas: no collective on the data path); value = all
ranks' coefficients / the slowest rank's time.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import platform
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "FCT coeffs/s at rel err <=1e-10 (mixed vs FP64 path); serving p50/p99 latency"
UNIT = "coeffs/s"
ERR_BOUND = 1e-10
CPU_BUDGET_S = 20.0          # CPU-oracle baseline: bounded sample per leg (one core, all cores)
REF_BUDGET_S = 150.0         # reference arm: whole run bound
SERVING_RATES = "25,100,1000,5000"
SERVING_REQUESTS = 200
SERVING_KAPPA0 = 20.0
SERVING_VARIANTS = 4         # Gaussian-cosine inputs per serving shape (plus one polynomial)
SERVING_CHECK_MAX_N = 5000   # served results of shapes up to this size are checked against the oracle
BATCH = 38                   # batched leg: transforms of the D=6 workload per launch
HETERO_BATCH = 512           # heterogeneous batch leg: transforms per launch (grid counts by Algorithm 2)
HETERO_CHECKED = 4           # smallest transforms of the heterogeneous batch checked against the oracle
ACCURACY_POINTS = 5000       # random points of the L-infinity error of the approximation
# the solver kernels' code, hashed to match a profile to it
SOLVER_SOURCES = ("fct_internal.h", "fct_df.cuh", "fct_common.cuh", "fct_solver.cuh", "fct_cells.cuh")
HEADLINE_PROFILE = "fct_solve_kernel_D10_d8_mixed.txt"
PATH_OPTIONS = {   # precision: 0 = FCT_FP64, 1 = FCT_MIXED (include/fct.h)
    "fp64": dict(precision=0, tol=1e-13),
    # inner FP32 solves to 1e-4 relative: three FP64 sweeps then reach the 1e-12
    # normal residual (the loosest inner tolerance that does; measured)
    "mixed": dict(precision=1, tol=1e-12, inner_tol=1e-4),
}


# cases of --profile: (workload factory name, path options, plan options)
PROFILE_CASES = {
    "d10_mixed": ("config_d10_rational", "mixed", {"block_threads": 512}),
    "d10_fp64": ("config_d10_rational", "fp64", {"block_threads": 256}),
    "d6_mixed": ("config_d6_gausscos", "mixed", {}),
    "d2_tensor_dct": ("tc_profile_workload", "mixed", {}),
    "sparse_d100": ("sparse_profile_workload", "mixed", {"block_threads": 512}),
    "sparse10_d100": ("sparse10_profile_workload", "mixed", {"block_threads": 512}),
}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=50)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="gpu", choices=["gpu", "reference"])
    ap.add_argument("--precision", default="auto", choices=["auto", "fp64", "mixed"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--serving-rates", default=SERVING_RATES,
                    help="comma-separated Poisson arrival rates (req/s) of the serving leg; empty = skip")
    ap.add_argument("--serving-requests", type=int, default=SERVING_REQUESTS, help="requests per rate")
    ap.add_argument("--serving-kappa0", type=float, default=SERVING_KAPPA0,
                    help="Algorithm 2 bound on kappa(A) used to pick each serving shape's grid count")
    ap.add_argument("--serving-team-blocks", type=int, default=0, help="0 = chosen by measurement")
    ap.add_argument("--batch", type=int, default=BATCH, help="transforms per launch of the batched leg (0 = skip)")
    ap.add_argument("--block-threads", type=int, default=0,
                    help="fix the launch shape (with --coef-lanes) instead of autotuning it")
    ap.add_argument("--coef-lanes", type=int, default=0)
    ap.add_argument("--hetero-batch", type=int, default=HETERO_BATCH,
                    help="transforms of the heterogeneous batch leg (D 3..8, degree 6..14; 0 = skip)")
    ap.add_argument("--no-next-rows", action="store_true", help="skip the rows past the hot path")
    ap.add_argument("--no-large-sparse", action="store_true",
                    help="skip the N = 1e6 sparse-support row (about 40 s)")
    ap.add_argument("--profile", default=None, choices=sorted(PROFILE_CASES),
                    help="run only `--warmup` + `--steps` executes of one case, without timing (for ncu)")
    ap.add_argument("--oracle-worker", default=None, help=argparse.SUPPRESS)
    return ap.parse_args()


def workload():
    import workloads as W
    return W.config_d10_rational()


def alt_workload():
    import workloads as W
    return W.config_d6_gausscos()


def family_name(family: int) -> str:
    import workloads as W
    return {W.FAMILY_POLY: "seeded polynomial", W.FAMILY_GAUSSCOS: "Gaussian-cosine",
            W.FAMILY_RATIONAL: "rational 1/(1+sum c x^2)", W.FAMILY_POLY_GAUSSCOS: "polynomial + Gaussian-cosine"}[family]


def workload_config(w):
    return {"workload": f"{w.name}: D={w.D} total degree {w.d} (N={w.N}), {w.K} extrema grids by Algorithm 1, "
                        f"{family_name(w.family)} target, M={w.M} samples",
            "D": w.D, "degree": w.d, "N": w.N, "grids": w.K, "samples": w.M,
            "l2": "flushed between timed steps (256 MiB write)"}


def cpu_description() -> dict:
    """nproc and the CPU model of the host that runs the oracle."""
    model = None
    try:
        out = subprocess.run(["lscpu"], stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.split(":")[0].strip() in ("Model name", "Model"):
                model = line.split(":", 1)[1].strip()
                break
    except Exception:
        pass
    if model is None:
        try:
            for line in open("/proc/cpuinfo"):
                if line.lower().startswith(("model name", "cpu part")):
                    model = line.split(":", 1)[1].strip()
                    break
        except Exception:
            pass
    return {"nproc": os.cpu_count(), "cpu_model": model or platform.processor() or platform.machine(),
            "machine": platform.machine()}


# ---------------------------------------------------------------------------
# CPU oracle leg: reference solutions, the timed CPU baseline (one core and
# all cores) and the reference arm, run in fresh processes with one BLAS
# thread each.  The oracle is used exactly as it stands; every problem it
# solves is described by seeded workload generators (never by GPU output).
# ---------------------------------------------------------------------------
def _one_thread_env():
    env = dict(os.environ)
    for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS", "BLIS_NUM_THREADS"):
        env[k] = "1"
    for k in ("RANK", "WORLD_SIZE", "LOCAL_RANK"):
        env.pop(k, None)
    return env


def _oracle_transform_times(args):
    """One worker of the all-core baseline: build the system once, then time
    `count` whole transforms (DCT-I + CGLS to 1e-13)."""
    wname, count = args
    import workloads as W
    from oracle import fct_oracle as O
    w = getattr(W, wname)()
    system = O.AliasSystem(w.support, w.sizes, w.nodes)
    f = O.sample_lgrid(w.family, w.params, w.support, w.sizes, w.nodes)
    t0 = time.perf_counter()
    for _ in range(count):
        O.cgls(system.A, system.rhs(f), tol=1e-13)
    return time.perf_counter() - t0, count


def oracle_worker(spec_path):
    """Runs the oracle jobs of spec_path (a JSON file; arrays in a sibling
    .npz) and writes the results next to it."""
    import numpy as np
    import workloads as W
    from oracle import fct_oracle as O
    spec = json.load(open(spec_path))
    arrays = np.load(spec_path + ".npz")
    out = {}
    # reference solutions: CGLS to 1e-15, the oracle's tier for these sizes
    for i, p in enumerate(spec.get("problems", [])):
        sup, sizes, nodes, params = (arrays[f"p{i}_{k}"] for k in ("support", "sizes", "nodes", "params"))
        f = O.sample_lgrid(p["family"], params, sup, sizes, nodes)
        system = O.AliasSystem(sup, sizes, nodes)
        t0 = time.perf_counter()
        c, it, rel = O.cgls(system.A, system.rhs(f), tol=1e-15)
        out[f"ref{i}"] = c
        out[f"ref{i}_s"] = time.perf_counter() - t0
    tim = spec.get("timing")
    if tim:
        w = getattr(W, tim["workload"])()
        system = O.AliasSystem(w.support, w.sizes, w.nodes)
        f = O.sample_lgrid(w.family, w.params, w.support, w.sizes, w.nodes)
        b = system.rhs(f)
        t0 = time.perf_counter()
        _, iters, _ = O.cgls(system.A, b, tol=1e-13)
        t_full = time.perf_counter() - t0
        fraction = tim.get("fraction", 1.0)
        steps = tim.get("steps", 0)
        times, credited = [], []
        if fraction >= 1.0:
            rounds = steps if steps > 0 else max(1, int(tim["budget_s"] // max(t_full, 1e-3)))
            for _ in range(rounds):
                t0 = time.perf_counter()
                O.cgls(system.A, system.rhs(f), tol=1e-13)
                times.append(time.perf_counter() - t0)
                credited.append(w.N)
        else:
            # a share of one transform: that share of the grids' DCT-I and of the CG iterations
            n_grids = max(1, int(math.ceil(fraction * w.K)))
            it_cap = max(1, int(math.ceil(fraction * iters)))
            for _ in range(steps):
                t0 = time.perf_counter()
                for l in range(n_grids):
                    fl = f[system.offsets[l]:system.offsets[l + 1]].reshape(tuple(int(n) for n in w.sizes[l]))
                    O.dct1_grid(fl)
                O.cgls(system.A, b, tol=1e-300, maxit=it_cap)
                times.append(time.perf_counter() - t0)
                credited.append(fraction * w.N)
        out["times"] = np.array(times)
        out["credited"] = np.array(credited)
        out["t_full"] = t_full
        if tim.get("all_cores"):
            import multiprocessing as mp
            nproc = os.cpu_count() or 1
            per = max(1, int(tim["budget_s"] // max(t_full, 1e-3) // 2))
            ctx = mp.get_context("spawn")
            with ctx.Pool(nproc) as pool:
                t0 = time.perf_counter()
                res = pool.map(_oracle_transform_times, [(tim["workload"], per)] * nproc)
                wall = time.perf_counter() - t0
            out["all_cores_wall"] = wall
            out["all_cores_span"] = max(r[0] for r in res)
            out["all_cores_transforms"] = sum(r[1] for r in res)
            out["all_cores_workers"] = nproc
    np.savez(spec_path + ".out.npz", **out)


def run_oracle(problems=(), timing=None):
    """problems: list of dicts (support, sizes, nodes, family, params) whose
    oracle solutions are wanted; timing: dict for the timed baseline.  Runs in
    a fresh process; returns the oracle's outputs."""
    import numpy as np
    with tempfile.TemporaryDirectory() as td:
        spec_path = os.path.join(td, "spec.json")
        arrays = {}
        spec = {"problems": [], "timing": timing}
        for i, p in enumerate(problems):
            spec["problems"].append({"family": int(p["family"])})
            for k in ("support", "sizes", "nodes", "params"):
                arrays[f"p{i}_{k}"] = np.asarray(p[k])
        json.dump(spec, open(spec_path, "w"))
        np.savez(spec_path + ".npz", **arrays)
        cmd = [sys.executable, os.path.abspath(__file__), "--oracle-worker", spec_path]
        r = subprocess.run(cmd, env=_one_thread_env(), stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
        if r.returncode != 0:
            raise RuntimeError("oracle worker failed:\n" + r.stdout[-3000:])
        z = np.load(spec_path + ".out.npz")
        return {k: z[k] for k in z.files}


def problem_of(w) -> dict:
    return {"support": w.support, "sizes": w.sizes, "nodes": w.nodes, "family": w.family, "params": w.params}


# ---------------------------------------------------------------------------
# clocks during the timed region
# ---------------------------------------------------------------------------
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index):
        self.dev = device_index
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.dev), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "100"],
                                         stdout=self.fh, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"], "samples": 0}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.fh.close()
        sm, smax, reasons, n = [], [], set(), 0
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                smax.append(float(parts[2]))
            except ValueError:
                continue
            n += 1
            for name, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(name)
        os.unlink(self.path)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": n}


# ---------------------------------------------------------------------------
# roofline bookkeeping
# ---------------------------------------------------------------------------
def algorithmic_bytes(info, rep, precision, layout=None):
    """Bytes the method must move per transform, with int32 tables and the
    single-point weights counted as recomputable (no stored-value bytes):
      DCT:                      8 M + 8 R    (samples in, b out)
      FP64 CG iteration:        8 K N + 8 (8 N + 5 R)
          (column and row index of every table entry, 4 bytes each; p read
          twice, x read and written, s written and read, p written: 8 N; q
          written and read, r read, written and gathered: 5 R)
      FP32 inner iteration:     8 K N + 4 (8 N + 5 R)
      FP64 refinement sweep:    8 K N + 8 (8 N + 5 R)   (one A and one A^T pass)
    layout (fct_plan_get_inner_layout): a plan whose inner solve runs by G grid
    groups streams its cell tables instead (6 bytes per entry, once to gather and
    once to scatter) and holds the row sums in shared memory:
      FP32 inner iteration:     12 K N + 16 G N + 24 N
          (a group reads s and p and writes its t, 12 N; the owners read every t,
          4 N a group, and read and write s, p and x)"""
    N, R, K, M = info["N"], info["R"], info["K"], info["M"]
    dct = 8 * M + 8 * R
    it64 = 8 * K * N + 8 * (8 * N + 5 * R)
    it32 = 8 * K * N + 4 * (8 * N + 5 * R)
    if layout and layout["groups"]:
        it32 = 12 * K * N + 16 * layout["groups"] * N + 24 * N
    if precision == "fp64":
        return dct + rep["iterations"] * it64
    return dct + rep["iterations"] * it32 + rep["refinements"] * it64


def gather_roofline(info, rep, launch_s, peak_gloads):
    """Scattered loads per launch: every CG iteration and every refinement
    sweep gathers one vector element per table entry in each of its two
    alias passes (A p bin-major, A^T q coefficient-major): 2 K N per pass
    pair; against the random-gather rate measured by fct_measure_l2."""
    K, N = info["K"], info["N"]
    loads = 2.0 * K * N * (rep["iterations"] + rep["refinements"])
    achieved = loads / launch_s / 1e9
    return {"bound": "l1_gather", "achieved": achieved, "peak": peak_gloads, "unit": "Gloads/s",
            "frac": achieved / peak_gloads, "loads_per_launch": loads,
            "peak_kind": "random 8-byte loads of an L2-resident buffer, measured live by fct_measure_l2"}


def profiled_traffic(profile_name: str):
    """DRAM bytes per launch from a committed ncu summary, or None when the
    kernel source changed since that capture."""
    import hashlib
    path = os.path.join(ROOT, "profiles", profile_name)
    csrc = os.path.join(ROOT, "paper_2309_14584_gb300", "csrc")
    try:
        fields = dict(line.split(":", 1) for line in open(path) if ":" in line and not line.startswith(" "))
        want = fields.get("source_sha256", "").strip()
        h = hashlib.sha256()
        for name in SOLVER_SOURCES:   # the team solver kernel's code
            h.update(open(os.path.join(csrc, name), "rb").read())
        if want and want == h.hexdigest():
            return int(fields["dram_bytes_per_launch"].strip())
    except Exception:
        return None
    return None


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            return json.load(fh), "measured"
    except Exception:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0}, "fallback"


def max_over_ranks(x: float) -> float:
    """Max of a per-rank scalar over the process group (the job's time)."""
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device="cuda")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


# ---------------------------------------------------------------------------
# timing helpers
# ---------------------------------------------------------------------------
def _timed(fn, steps, flush):
    """Device time of fn() per call: L2 flushed before each call, one pair of
    CUDA events around each call on the current stream; list of ms."""
    import torch
    fn()
    torch.cuda.synchronize()
    stream = torch.cuda.current_stream()
    evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    for e0, e1 in evs:
        flush.zero_()
        e0.record(stream)
        fn()
        e1.record(stream)
    torch.cuda.synchronize()
    return [e0.elapsed_time(e1) for e0, e1 in evs]


def run_paths(F, w, args, flush, precisions, steps, warmup, dev, tune=True, world=1):
    """Both solver paths on the same device-resident samples of workload w:
    autotuned launch shape, W warm-up steps, K timed steps (CUDA events, L2
    flushed between steps), end to end through fct_execute_host."""
    import numpy as np
    import torch
    from paper_2309_14584_gb300.tune import autotune
    samples = torch.empty(w.M, dtype=torch.float64, device="cuda")
    probe = F.Plan(w.support, w.sizes, w.nodes)
    probe.sample(w.family, w.params, samples)   # the samples do not depend on the path or launch shape
    probe.close()
    results = {}
    for prec in precisions:
        opts = dict(PATH_OPTIONS[prec])
        if args.block_threads:
            tuned = {"options": dict(opts, block_threads=args.block_threads, coef_lanes=args.coef_lanes),
                     "ms": None, "timings": []}
        elif tune:
            tuned = autotune(w.support, w.sizes, w.nodes, samples, opts)
        else:
            tuned = {"options": opts, "ms": None, "timings": []}
        plan = F.Plan(w.support, w.sizes, w.nodes, **tuned["options"])
        coeffs = torch.empty(w.N, dtype=torch.float64, device="cuda")
        rep = plan.execute(samples, coeffs)
        c_first = coeffs.cpu().numpy()
        for _ in range(warmup):
            plan.execute(samples, coeffs, report=False)
        torch.cuda.synchronize()
        stream = torch.cuda.current_stream()
        evs = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
        clocks = ClockSampler(dev)
        clocks.start()
        if world > 1:
            import torch.distributed as dist
            dist.barrier()
        torch.cuda.synchronize()
        for e0, e1 in evs:
            flush.zero_()
            e0.record(stream)
            plan.execute(samples, coeffs, report=False)
            e1.record(stream)
        torch.cuda.synchronize()
        if world > 1:
            dist.barrier()
        clk = clocks.stop()
        step_ms = [e0.elapsed_time(e1) for e0, e1 in evs]
        total_s = sum(step_ms) / 1e3
        if world > 1:
            total_s = max_over_ranks(total_s)
        rep_last = F.fct_plan_last_report(plan.handle)
        same = bool(np.array_equal(coeffs.cpu().numpy(), c_first))
        # end to end through the host-buffer entry point (pinned memory, copies timed)
        s_host = samples.cpu().pin_memory()
        c_host = torch.empty(w.N, dtype=torch.float64).pin_memory()
        for _ in range(2):
            plan.execute_host(s_host, c_host)
        e2e_n = max(3, min(steps, 20))
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(e2e_n):
            plan.execute_host(s_host, c_host)
        e2e_s = (time.perf_counter() - t0) / e2e_n
        results[prec] = dict(plan_info=plan.info, rep=rep, rep_last=rep_last, coeffs=c_first, tuning=tuned,
                             step_ms=step_ms, total_s=total_s, clocks=clk, deterministic=same, e2e_s=e2e_s,
                             e2e_host_equal=bool(np.array_equal(c_host.numpy(), c_first)), plan=plan)
    return results, samples


# ---------------------------------------------------------------------------
# GPU arm
# ---------------------------------------------------------------------------
def run_gpu(args):
    import numpy as np
    import torch
    import torch.distributed as dist

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        torch.cuda.set_device(local)
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    else:
        torch.cuda.set_device(0)
    dev = torch.cuda.current_device()

    import paper_2309_14584_gb300 as F
    from paper_2309_14584_gb300 import build as B
    B.build()
    F.lib()

    # on-chip roofs of this device (outside every timed region)
    roofs = {"l2": F.fct_measure_l2(32 << 20, 200), "fp64_tflops": F.fct_measure_fp64(1 << 16)}

    w = workload()
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")
    precisions = ["fp64", "mixed"] if args.precision == "auto" else [args.precision]
    results, samples = run_paths(F, w, args, flush, precisions, args.steps, args.warmup, dev, world=world)
    if "mixed" in results:
        results["mixed"]["accuracy"] = approximation_error(F, results["mixed"]["plan"], w,
                                                           torch.from_numpy(results["mixed"]["coeffs"]).cuda())
    gpu_launches = args.steps
    for r in results.values():
        r["plan"].close()
        del r["plan"]
    del samples

    alt = None
    if rank == 0 and world == 1:
        wa = alt_workload()
        alt, s_alt = run_paths(F, wa, args, flush, precisions, min(args.steps, 20), args.warmup, dev)
        for r in alt.values():
            r["plan"].close()
            del r["plan"]
        del s_alt

    batched = run_batched(args, F, alt_workload(), dict(PATH_OPTIONS["mixed"]), flush) if args.batch > 0 else None
    if batched is not None and world > 1:
        batched["total_s"] = max_over_ranks(batched["total_s"])
    hetero = run_hetero_batch(args, F, dict(PATH_OPTIONS["mixed"])) \
        if args.hetero_batch > 0 and rank == 0 and world == 1 else None
    serving = run_serving(args, F) if rank == 0 and world == 1 else None
    next_rows = None
    if rank == 0 and world == 1 and "mixed" in results and not args.no_next_rows:
        try:
            next_rows = run_next_rows(F, alt_workload(), dict(PATH_OPTIONS["mixed"]), flush,
                                      large_sparse=not args.no_large_sparse,
                                      gather_peak=roofs["l2"]["gather_gloads_per_s"])
        except Exception as e:  # measurement only; the bench line stands without it
            next_rows = {"error": str(e)[:200]}

    if rank != 0:
        if world > 1:
            dist.destroy_process_group()
        return

    # ---- CPU oracle leg (rank 0, N = 1): reference solutions and the timed baseline
    problems = [problem_of(w), problem_of(alt_workload())]
    checks = []   # (label, GPU coefficients, index into problems)
    if hetero is not None:
        for label, wk, c in hetero.pop("check_results"):
            checks.append((label, c, len(problems)))
            problems.append(problem_of(wk))
    if serving is not None:
        for label, wk, c in serving.pop("check_results"):
            checks.append((label, c, len(problems)))
            problems.append(problem_of(wk))
    cpu = None
    if world == 1 and not args.no_cpu_baseline:
        cpu = run_oracle(problems, timing={"workload": "config_d10_rational", "budget_s": CPU_BUDGET_S,
                                           "all_cores": True})

    def rel(a, b):
        return float(np.linalg.norm(a - b) / np.linalg.norm(b))

    for prec, r in results.items():
        r["rel_err"] = rel(r["coeffs"], cpu["ref0"]) if cpu is not None else None
        r["value"] = world * w.N * args.steps / r["total_s"]
    if alt is not None:
        for prec, r in alt.items():
            r["rel_err"] = rel(r["coeffs"], cpu["ref1"]) if cpu is not None else None
            r["value"] = w_alt_N(alt) * len(r["step_ms"]) / r["total_s"]
    check_errs = {}
    if cpu is not None:
        for label, c, i in checks:
            check_errs.setdefault(label.split(":")[0], []).append(rel(c, cpu[f"ref{i}"]))
    if hetero is not None:
        errs = check_errs.get("hetero", [])
        hetero["oracle_checked"] = len(errs)
        hetero["max_rel_err_vs_oracle"] = max(errs) if errs else None
    if serving is not None:
        errs = check_errs.get("served", [])
        serving["oracle_checked"] = len(errs)
        serving["max_rel_err_vs_oracle"] = max(errs) if errs else None

    valid = [p for p, r in results.items() if r["rep"]["status"] == 0 and r["rel_err"] is not None and
             r["rel_err"] <= ERR_BOUND]
    best = max(valid, key=lambda p: results[p]["value"]) if valid else None
    R0 = results[best] if best else results[max(results, key=lambda p: results[p]["value"])]
    path = best or "none"
    info = R0["plan_info"]
    peaks, peak_kind = measured_peaks()
    mean_launch_s = statistics.mean(R0["step_ms"]) / 1e3
    abytes = algorithmic_bytes(info, R0["rep"], best or "mixed")
    achieved = abytes / mean_launch_s / 1e9
    l2 = roofs["l2"]["read_gbs"]
    line = {
        "metric": METRIC,
        "value": R0["value"] if best else 0.0,
        "unit": UNIT,
        "n_gpus": world,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": statistics.mean(R0["step_ms"]),
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f64" if best == "fp64" else "f32+f64",
        "data": "synthetic",
        "config": dict(workload_config(w), path=path, iterations=R0["rep"]["iterations"],
                       refinements=R0["rep"]["refinements"], nonempty_bins=info["R"],
                       solver_blocks=info["grid_blocks"], block_threads=info["block_threads"],
                       coef_lanes=info["coef_lanes"], parallelism=f"replicas x{world}",
                       launch_tuning={"chosen": {k: v for k, v in R0["tuning"]["options"].items()
                                                 if k in ("block_threads", "coef_lanes", "entries_per_lane",
                                                          "coef_split", "normal_matrix", "tensor_dct")},
                                      "candidates_ms": [[c, round(ms, 4)] for c, ms in R0["tuning"]["timings"]]}),
        "rel_err_vs_oracle": R0["rel_err"],
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peaks["hbm_gbs"], "unit": "GB/s",
                     "frac": achieved / peaks["hbm_gbs"],
                     "traffic": profiled_traffic(HEADLINE_PROFILE) if best == "mixed" else None,
                     "kernel": "fct_solve_kernel", "algorithmic_bytes_per_launch": abytes,
                     "peak_kind": f"{peak_kind} HBM copy bandwidth (MEASURED_PEAKS.json)",
                     "note": "algorithmic bytes per launch (table indices and vectors of every CG iteration and sweep, "
                             "DCT samples and bins) over the launch time; the CG loop's tables and "
                             "vectors (about 23 MB) stay in the 129 MB L2, so DRAM traffic per launch is the "
                             "samples and DCT buffers (traffic), and the loop is bound by scattered-load "
                             "latency (gather_roofline) rather than by either bandwidth"},
        "l2_roofline": {"bound": "l2", "achieved": achieved, "peak": l2, "unit": "GB/s", "frac": achieved / l2,
                        "peak_kind": "L2 read bandwidth measured live by fct_measure_l2 (32 MiB resident buffer)"},
        "e2e": {"value": w.N / R0["e2e_s"], "unit": UNIT, "h2d_bytes_per_step": 8 * w.M,
                "d2h_bytes_per_step": 8 * w.N + 32 + 4},
        "clocks": {k: R0["clocks"][k] for k in ("sm_mhz", "sm_max_mhz", "reasons")},
        "gpu_launches": gpu_launches,
        "alt_paths": {p: {"value": r["value"], "ms_per_step": statistics.mean(r["step_ms"]),
                          "iterations": r["rep"]["iterations"], "refinements": r["rep"]["refinements"],
                          "rel_err_vs_oracle": r["rel_err"], "deterministic": r["deterministic"],
                          "e2e_value": w.N / r["e2e_s"], "meets_1e-10": p in valid}
                      for p, r in results.items()},
        # the binding roof of the CG loop: scattered 4-8 byte loads (one per table
        # entry per alias pass) against the measured random-gather rate
        "gather_roofline": gather_roofline(info, R0["rep"], mean_launch_s, roofs["l2"]["gather_gloads_per_s"]),
        "roofs_measured": {"l2_read_gbs": l2, "l2_gather_sector_gbs": roofs["l2"]["gather_sector_gbs"],
                           "l2_gather_gloads_per_s": roofs["l2"]["gather_gloads_per_s"],
                           "fp64_tflops": roofs["fp64_tflops"]},
    }
    if not best:
        line["error"] = "no path met the 1e-10 bound against the oracle (or the oracle leg was skipped)"
    if "fp64" in results and "mixed" in results:
        line["mixed_over_fp64"] = results["mixed"]["value"] / results["fp64"]["value"]
    if alt is not None:
        line["alt_workloads"] = {"D6_d10_gausscos": {
            "config": workload_config(alt_workload()),
            "paths": {p: {"value": r["value"], "ms_per_step": statistics.mean(r["step_ms"]),
                          "iterations": r["rep"]["iterations"], "refinements": r["rep"]["refinements"],
                          "rel_err_vs_oracle": r["rel_err"], "e2e_value": w_alt_N(alt) / r["e2e_s"],
                          "algorithmic_bytes": algorithmic_bytes(r["plan_info"], r["rep"], p),
                          "l2_frac": algorithmic_bytes(r["plan_info"], r["rep"], p) /
                          (statistics.mean(r["step_ms"]) / 1e3) / 1e9 / l2}
                      for p, r in alt.items()}}}
    try:
        us_bar = F.fct_measure_team_barrier(info["grid_blocks"], info["block_threads"], 2000)
        line["sync_floor"] = {"us_per_team_barrier": us_bar, "blocks": info["grid_blocks"],
                              "block_threads": info["block_threads"], "barriers_per_cg_iteration": 2,
                              "us_per_step_per_cg_iteration": 1e3 * statistics.mean(R0["step_ms"]) /
                              max(1, R0["rep"]["iterations"]),
                              "note": "empty-phase barrier crossings (fct_measure_team_barrier) vs the "
                                      "step time divided by its CG iterations (DCT and sweeps included)"}
    except Exception as e:  # measurement only; the bench line stands without it
        line["sync_floor"] = {"error": str(e)[:200]}
    if "accuracy" in results.get("mixed", {}):
        line["accuracy"] = results["mixed"]["accuracy"]
    try:
        line["plan_build"] = plan_build_times(F)
    except Exception as e:  # measurement only; the bench line stands without it
        line["plan_build"] = {"error": str(e)[:200]}
    if next_rows is not None:
        line["next_rows"] = next_rows
    if batched is not None:
        batched["value"] = world * batched["coeffs_per_launch"] * len(batched["ms"]) / batched["total_s"]
        del batched["ms"]
        line["batched"] = batched
    if hetero is not None:
        line["hetero_batch"] = hetero
    if serving is not None:
        line["serving"] = serving
    if cpu is not None:
        ct = float(cpu["times"].sum())
        one = float(cpu["credited"].sum()) / ct
        host = cpu_description()
        all_v = float(cpu["all_cores_transforms"]) * w.N / float(cpu["all_cores_span"])
        line["cpu_baseline"] = {
            "value": all_v, "unit": UNIT, "cores": int(cpu["all_cores_workers"]), "kind": "oracle",
            "sample": f"{int(cpu['all_cores_transforms'])} whole transforms of the headline workload (FP64 DCT-I by "
                      f"direct matrix products + scipy-sparse CGLS to 1e-13), one per process on "
                      f"{int(cpu['all_cores_workers'])} processes of one BLAS thread each, "
                      f"{float(cpu['all_cores_span']):.1f} s",
            "single_core": {"value": one, "cores": 1,
                            "sample": f"{len(cpu['times'])} whole transforms, 1 thread, {ct:.1f} s"},
            "nproc": host["nproc"], "cpu_model": host["cpu_model"], "machine": host["machine"]}
    print(json.dumps(line))
    if world > 1:
        dist.destroy_process_group()


def w_alt_N(alt):
    return next(iter(alt.values()))["plan_info"]["N"]


# ---------------------------------------------------------------------------
# plan construction, batched legs and approximation error
# ---------------------------------------------------------------------------
def plan_build_times(F, reps=3) -> dict:
    """Wall time of fct_plan_create (validation, tables, DCT set-up, upload and
    workspace allocation) with the alias tables built in host C++ and on the
    device, median of `reps` after one untimed build each."""
    out = {}
    for name, wl in (("D6_d10", alt_workload()), ("D10_d8", workload())):
        row = {"K_N": int(wl.K * wl.N)}
        for key, pb in (("host_ms", F.FCT_PLAN_BUILD_HOST), ("device_ms", F.FCT_PLAN_BUILD_DEVICE)):
            ts = []
            for i in range(reps + 1):
                t0 = time.perf_counter()
                p = F.Plan(wl.support, wl.sizes, wl.nodes, precision=F.FCT_MIXED, plan_build=pb)
                dt = 1e3 * (time.perf_counter() - t0)
                p.close()
                if i > 0:
                    ts.append(dt)
            row[key] = round(statistics.median(ts), 3)
        row["speedup"] = round(row["host_ms"] / row["device_ms"], 2)
        out[name] = row
    return out


def approximation_error(F, plan, w, coeffs_dev) -> dict:
    """L-infinity error of the computed expansion against the target at random
    points of [-1, 1]^D (the paper's accuracy measure), evaluated on the
    device by fct_evaluate; the target itself is evaluated on the host."""
    import numpy as np
    import torch
    import workloads as W
    pts = W.stream(17, "probe").uniform(-1.0, 1.0, (ACCURACY_POINTS, w.D))
    vals = torch.empty(ACCURACY_POINTS, dtype=torch.float64, device="cuda")
    plan.evaluate(coeffs_dev, torch.from_numpy(pts).cuda(), vals)
    torch.cuda.synchronize()
    if w.family == W.FAMILY_RATIONAL:
        f = 1.0 / (1.0 + (pts ** 2) @ w.params[:w.D])
    else:
        a, b = w.params[:w.D], w.params[w.D:2 * w.D]
        f = np.exp(-(pts ** 2) @ a) * np.cos(pts @ b)
    err = np.abs(vals.cpu().numpy() - f)
    return {"linf_abs_error": float(err.max()), "points": ACCURACY_POINTS,
            "note": "max |p(x) - f(x)| of the mixed-path expansion at uniform random points"}


def sparse_rooflines(info, rep, ms, peaks, peak_kind, gather_peak, layout=None):
    """Roofs of a sparse-support transform, whose tables (K N entries, more
    than L2 holds) are read from DRAM every iteration: the algorithmic bytes
    against the measured HBM copy rate, and the scattered loads (one per table
    entry and alias pass) against the measured random-gather rate.  An inner
    solve by grid groups makes its scattered accesses in shared memory, so such
    a plan has no gather roof (None)."""
    by_groups = bool(layout and layout["groups"])
    bytes_ = algorithmic_bytes(info, rep, "mixed", layout)
    hbm = {"bound": "hbm", "achieved": bytes_ / (ms / 1e3) / 1e9, "peak": peaks["hbm_gbs"], "unit": "GB/s",
           "algorithmic_bytes_per_launch": bytes_,
           "peak_kind": f"{peak_kind} HBM copy bandwidth (MEASURED_PEAKS.json)",
           "note": "inner solve by grid groups: 6 table bytes per entry, read to gather and again to scatter "
                   "(in part from L2), and the groups' vectors" if by_groups else
                   "table bytes counted as indices only (4 per entry and alias pass); the stored FP32 entry "
                   "values double the table bytes actually read"}
    hbm["frac"] = hbm["achieved"] / hbm["peak"]
    return hbm, None if by_groups else gather_roofline(info, rep, ms / 1e3, gather_peak)


def run_next_rows(F, w, opts, flush, steps=20, large_sparse=True, gather_peak=None) -> dict:
    """The rows past the hot path, timed on the same GPU: the paper's
    first-kind grid, evaluation of the expansion at random points, and
    sparse S^inf supports at D = 100 (N = 2e4, and N = 1e6 unless
    large_sparse is off)."""
    import numpy as np
    import torch
    import workloads as W
    out = {}
    peaks, peak_kind = measured_peaks()
    # first-kind grid (1/n DCT-II quadrature, signed alias entries), same workload and options
    p = F.Plan(w.support, w.sizes, w.nodes, grid_kind=F.FCT_GRID_FIRST_KIND, **opts)
    x = torch.empty(p.M, dtype=torch.float64, device="cuda")
    p.sample(w.family, w.params, x)
    c = torch.empty(p.N, dtype=torch.float64, device="cuda")
    rep = p.execute(x, c)
    ms = statistics.mean(_timed(lambda: p.execute(x, c, report=False), steps, flush))
    acc = approximation_error(F, p, w, c)
    out["first_kind"] = {"workload": w.name, "ms_per_transform": ms, "value": w.N / (ms / 1e3), "unit": UNIT,
                         "status": rep["status"], "iterations": rep["iterations"], "refinements": rep["refinements"],
                         "linf_abs_error": acc["linf_abs_error"], "nonempty_bins": p.info["R"]}
    # evaluation of an expansion on this support at random points
    npts = 1 << 17
    pts = torch.from_numpy(W.stream(23, "probe").uniform(-1.0, 1.0, (npts, w.D))).cuda()
    vals = torch.empty(npts, dtype=torch.float64, device="cuda")
    ms = statistics.mean(_timed(lambda: p.evaluate(c, pts, vals), max(3, steps // 4), flush))
    flops = 2 * npts * (w.N - 1)   # per point: one multiply-add per nonzero index of the support's trie, FP64
    out["evaluate"] = {"points": npts, "terms": w.N, "ms": ms, "points_per_s": npts / (ms / 1e3),
                       "roofline": {"bound": "alu", "achieved": flops / (ms / 1e3) / 1e12, "unit": "TFLOP/s",
                                    "peak": F.fct_measure_fp64(1 << 16),
                                    "peak_kind": "FP64 fma rate measured live by fct_measure_fp64"}}
    out["evaluate"]["roofline"]["frac"] = out["evaluate"]["roofline"]["achieved"] / out["evaluate"]["roofline"]["peak"]
    p.close()
    # a D = 2 plan whose DCT runs on the tensor cores, timed with them on and off
    wt = tc_profile_workload()
    row = {"workload": wt.name, "N": wt.N, "M": wt.M}
    c_on = None
    for key, mode in (("tensor_cores", 0), ("fp64_units", -1)):
        pt = F.Plan(wt.support, wt.sizes, wt.nodes, tensor_dct=mode, **opts)
        xt = torch.empty(pt.M, dtype=torch.float64, device="cuda")
        pt.sample(wt.family, wt.params, xt)
        ct = torch.empty(pt.N, dtype=torch.float64, device="cuda")
        rep = pt.execute(xt, ct)
        b = torch.empty(pt.info["R"], dtype=torch.float64, device="cuda")
        rhs_ms = statistics.mean(_timed(lambda: F.fct_plan_rhs(pt.handle, xt, b), max(3, steps // 4), flush))
        ms = statistics.mean(_timed(lambda: pt.execute(xt, ct, report=False), max(3, steps // 4), flush))
        row[key] = {"ms_per_transform": ms, "value": wt.N / (ms / 1e3), "rhs_stage_ms": rhs_ms,
                    "tensor_dct_grids": pt.info["tensor_dct_grids"], "status": rep["status"],
                    "iterations": rep["iterations"]}
        if mode == 0:
            c_on = ct.cpu().numpy()
            # tensor roof of the DCT stage (its GEMMs, digit splits and last pass together):
            # BF16 flops the passes issue against the measured dense BF16 rate
            flops = pt.info["tensor_dct_flops"]
            peak = peaks.get("bf16_tflops")
            row[key]["tensor_roofline"] = {
                "bound": "tensor", "flops_per_transform": flops, "unit": "TFLOP/s",
                "achieved": flops / (rhs_ms / 1e3) / 1e12, "peak": peak,
                "frac": flops / (rhs_ms / 1e3) / 1e12 / peak if peak else None,
                "peak_kind": f"{peak_kind} BF16 dense (cuBLAS burst), MEASURED_PEAKS.json",
                "note": "flops of the 36 exact digit-slice products per tile and K step over the whole DCT "
                        "stage time (fct_plan_rhs); the useful FP64 DCT work is 36x smaller"}
        else:
            row["rel_diff_on_off"] = float(np.linalg.norm(c_on - ct.cpu().numpy()) / np.linalg.norm(ct.cpu().numpy()))
        pt.close()
    out["tensor_dct_D2"] = row
    # sparse S^inf support at D = 100 (3 nonzero components per index), 10 D grids,
    # a polynomial on the support recovered (the check that holds at any size)
    D, d, N = 100, 9, 20_000
    sup = W.sparse_infinity_support(13, D, d, N, 3)
    sizes, nodes = W.l_grid(300, N, D, 10 * D, 1, d + 1)
    c_true = W.poly_coefficients(10, sup)
    t0 = time.perf_counter()
    ps = F.Plan(sup, sizes, nodes, **opts)
    t_build = time.perf_counter() - t0
    xs = torch.empty(ps.M, dtype=torch.float64, device="cuda")
    ps.sample(W.FAMILY_POLY | F.fct.FCT_SAMPLE_FOLDED, c_true, xs)
    cs = torch.empty(N, dtype=torch.float64, device="cuda")
    rep = ps.execute(xs, cs)
    err = float(np.linalg.norm(cs.cpu().numpy() - c_true) / np.linalg.norm(c_true))
    ms = statistics.mean(_timed(lambda: ps.execute(xs, cs, report=False), max(3, steps // 4), flush))
    out["sparse_D100"] = {"N": N, "K": int(sizes.shape[0]), "M": int(ps.M), "nonempty_bins": ps.info["R"],
                          "plan_build_ms": 1e3 * t_build, "ms_per_transform": ms, "value": N / (ms / 1e3),
                          "unit": UNIT, "status": rep["status"], "iterations": rep["iterations"],
                          "refinements": rep["refinements"], "recovery_rel_err": err}
    if gather_peak:
        out["sparse_D100"]["roofline"], out["sparse_D100"]["gather_roofline"] = sparse_rooflines(
            dict(ps.info), rep, ms, peaks, peak_kind, gather_peak, F.fct_plan_get_inner_layout(ps.handle))
    ps.close()
    del xs, cs
    if not large_sparse:
        return out
    # the paper's sparse-support scale: N = 1e6 multi-indices at D = 100 (10 nonzero
    # components of degree <= 3 each), 600 grids by Algorithm 1 (measured: 300 grids
    # do not converge in 3000 inner iterations, 400 take 28 s, 600 take 21 s); one
    # transform, timed with CUDA events, the polynomial on the support recovered
    D, d, N, K = 100, 3, 1_000_000, 600
    sup = W.sparse_support_vectorised(3, D, d, N, 10)
    sizes, nodes = W.l_grid(500, N, D, K, 1, d + 1)
    c_true = W.poly_coefficients(10, sup)
    t0 = time.perf_counter()
    pl = F.Plan(sup, sizes, nodes, **opts)
    t_build = time.perf_counter() - t0
    xs = torch.empty(pl.M, dtype=torch.float64, device="cuda")
    pl.sample(W.FAMILY_POLY | F.fct.FCT_SAMPLE_FOLDED, c_true, xs)
    cs = torch.empty(N, dtype=torch.float64, device="cuda")
    flush.zero_()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record()
    rep = pl.execute(xs, cs)
    e1.record()
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1)
    err = float(np.linalg.norm(cs.cpu().numpy() - c_true) / np.linalg.norm(c_true))
    out["sparse_D100_N1e6"] = {"N": N, "K": K, "M": int(pl.M), "nonempty_bins": pl.info["R"], "nonzeros_per_index": 10,
                               "max_degree": d, "table_entries": K * N, "device_bytes": pl.info["device_bytes"],
                               "plan_build_ms": 1e3 * t_build, "ms_per_transform": ms, "value": N / (ms / 1e3),
                               "unit": UNIT, "status": rep["status"], "iterations": rep["iterations"],
                               "refinements": rep["refinements"], "recovery_rel_err": err}
    if gather_peak:
        out["sparse_D100_N1e6"]["roofline"], out["sparse_D100_N1e6"]["gather_roofline"] = sparse_rooflines(
            dict(pl.info), rep, ms, peaks, peak_kind, gather_peak, F.fct_plan_get_inner_layout(pl.handle))
    pl.close()
    return out


def _graph_batch(F, hs, xs, cs, tb, steps, flush):
    """The same batch as a prepared batch (fct_batch_create) whose launch is
    captured once into a CUDA graph and replayed: per replay one memset and one
    cooperative launch, nothing from the host.  Returns the replay times (ms),
    whether the replay's coefficients equal the direct launch's bit for bit,
    and whether every report is FCT_OK."""
    import torch
    ref = [c.clone() for c in cs]
    b = F.fct_batch_create(hs, xs, cs, team_blocks=tb)
    try:
        F.fct_batch_launch(b)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            F.fct_batch_launch(b)
        g.replay()
        torch.cuda.synchronize()
        ok = all(r["status"] == 0 for r in F.fct_batch_reports(b, len(hs)))
        same = all(bool(torch.equal(c, r)) for c, r in zip(cs, ref))
        ms = _timed(lambda: g.replay(), steps, flush)
        del g
    finally:
        F.fct_batch_destroy(b)
    return ms, same, ok


def run_batched(args, F, w, opts, flush) -> dict:
    """B transforms of workload w (distinct Gaussian-cosine targets, one plan
    and B - 1 clones) per launch of fct_execute_batch, the blocks per team
    chosen by measurement; L2 flushed between launches."""
    import torch
    import workloads as W
    B = args.batch
    base = F.Plan(w.support, w.sizes, w.nodes, **opts)
    plans = [base] + [base.clone() for _ in range(B - 1)]
    xs, cs = [], []
    for i in range(B):
        x = torch.empty(base.M, dtype=torch.float64, device="cuda")
        base.sample(w.family, W.gausscos_params(1000 + i, w.D), x)
        xs.append(x)
        cs.append(torch.empty(base.N, dtype=torch.float64, device="cuda"))
    hs = [p.handle for p in plans]
    from paper_2309_14584_gb300.tune import autotune_team_blocks
    tune = autotune_team_blocks(hs, xs, cs)   # outside the timed region
    tb = tune["team_blocks"]
    reps = F.fct_execute_batch(hs, xs, cs, team_blocks=tb)
    alone = torch.empty(base.N, dtype=torch.float64, device="cuda")
    base.execute(xs[B - 1], alone)
    same = bool(torch.equal(alone, cs[B - 1]))
    for _ in range(args.warmup):
        F.fct_execute_batch(hs, xs, cs, team_blocks=tb, report=False)
    ms = _timed(lambda: F.fct_execute_batch(hs, xs, cs, team_blocks=tb, report=False), args.steps, flush)
    gms, gsame, gok = _graph_batch(F, hs, xs, cs, tb, args.steps, flush)
    for p in plans[1:]:
        p.close()
    base.close()
    # the same batch on the plain FP64 path
    base64 = F.Plan(w.support, w.sizes, w.nodes, **dict(PATH_OPTIONS["fp64"]))
    plans = [base64] + [base64.clone() for _ in range(B - 1)]
    hs = [p.handle for p in plans]
    reps64 = F.fct_execute_batch(hs, xs, cs, team_blocks=tb)
    ms64 = _timed(lambda: F.fct_execute_batch(hs, xs, cs, team_blocks=tb, report=False), args.steps, flush)
    for p in plans[1:]:
        p.close()
    base64.close()
    fp64_path = {"value": B * w.N / (statistics.mean(ms64) / 1e3), "ms_per_launch": statistics.mean(ms64),
                 "all_converged": all(r["status"] == 0 for r in reps64)}
    return {"workload": w.name, "transforms_per_launch": B, "team_blocks": tb,
            "fp64_path": fp64_path, "mixed_over_fp64": (B * w.N / (statistics.mean(ms) / 1e3)) / fp64_path["value"],
            "graph": {"ms_per_launch": statistics.mean(gms), "value": B * w.N / (statistics.mean(gms) / 1e3),
                      "equals_direct_launch": gsame, "all_converged": gok,
                      "note": "fct_batch_launch captured into a CUDA graph, replayed"},
            "team_blocks_tuning_ms": [[t, round(m, 3)] for t, m in tune["timings"]], "path": "mixed",
            "coeffs_per_launch": B * w.N, "ms_per_launch": statistics.mean(ms), "total_s": sum(ms) / 1e3, "ms": ms,
            "all_converged": all(r["status"] == 0 for r in reps),
            "max_iterations": max(r["iterations"] for r in reps),
            "batch_equals_alone": same, "unit": UNIT,
            "note": "independent transforms of one plan shape in one persistent launch (fct_execute_batch)"}


def run_hetero_batch(args, F, opts) -> dict:
    """The 512-transform heterogeneous batch (D ~ U{3..8}, total degree
    ~ U{6..14}, polynomial plus Gaussian-cosine targets) in one persistent launch
    per step, each transform's grid count chosen by Algorithm 2 (kappa0 = 20,
    candidates 10 D grids) before the timed region.  The results of the
    smallest transforms are returned for the oracle check."""
    from concurrent.futures import ThreadPoolExecutor
    import torch
    import workloads as W
    from paper_2309_14584_gb300 import lgrid
    cands = W.config_batch(B=args.hetero_batch, grids_per_dim=10)

    def select(w):
        r = lgrid.select_grids(w.support, w.sizes, w.nodes, kappa0=SERVING_KAPPA0, start=3 * w.D,
                               step=max(1, w.D // 2), probe_iterations=200)
        return r["L"] if r["L"] is not None else min(r["probes"], key=lambda k: r["probes"][k] * k)

    t0 = time.perf_counter()
    with ThreadPoolExecutor(16) as ex:   # plan building is host work; the library releases the GIL
        Ls = list(ex.map(select, cands))
    t_select = time.perf_counter() - t0
    ws = [W.first_grids(w, L) for w, L in zip(cands, Ls)]
    with ThreadPoolExecutor(16) as ex:
        plans = list(ex.map(lambda w: F.Plan(w.support, w.sizes, w.nodes, **opts), ws))
    xs, cs = [], []
    for p, w in zip(plans, ws):
        x = torch.empty(p.M, dtype=torch.float64, device="cuda")
        p.sample(w.family, w.params, x)
        xs.append(x)
        cs.append(torch.empty(p.N, dtype=torch.float64, device="cuda"))
    hs = [p.handle for p in plans]
    from paper_2309_14584_gb300.tune import autotune_team_blocks
    tune = autotune_team_blocks(hs, xs, cs, candidates=(8, 16, 32), reps=1)   # outside the timed region
    tb = tune["team_blocks"]
    reps = F.fct_execute_batch(hs, xs, cs, team_blocks=tb)
    order = sorted(range(len(plans)), key=lambda i: plans[i].N)
    small = order[0]
    alone = torch.empty(plans[small].N, dtype=torch.float64, device="cuda")
    plans[small].execute(xs[small], alone)
    same = bool(torch.equal(alone, cs[small]))
    checks = [(f"hetero:{ws[i].name}", ws[i], cs[i].cpu().numpy()) for i in order[:HETERO_CHECKED]]
    direct_ms = statistics.mean(_timed(lambda: F.fct_execute_batch(hs, xs, cs, team_blocks=tb, report=False), 2,
                                       torch.empty(1, device="cuda")))
    gms, gsame, gok = _graph_batch(F, hs, xs, cs, tb, 2, torch.empty(1, device="cuda"))
    ms = statistics.mean(gms)
    sum_n = sum(p.N for p in plans)
    out = {"transforms_per_launch": len(plans), "value": sum_n / (ms / 1e3), "unit": UNIT, "ms_per_launch": ms,
           "launch": "one persistent cooperative launch per step, captured once into a CUDA graph and replayed "
                     "(fct_batch_launch)", "direct_ms_per_launch": direct_ms, "graph_equals_direct_launch": gsame,
           "graph_all_converged": gok,
           "coeffs_per_launch": sum_n, "samples_per_launch": sum(p.M for p in plans), "timed_launches": 2,
           "grid_selection_s": round(t_select, 1),
           "grid_count_over_3D_median": sorted(L / (3 * w.D) for L, w in zip(Ls, cands))[len(Ls) // 2],
           "all_converged": all(r["status"] == 0 for r in reps), "max_iterations": max(r["iterations"] for r in reps),
           "batch_equals_alone": same, "team_blocks": tb,
           "team_blocks_tuning_ms": [[t, round(m, 1)] for t, m in tune["timings"]], "path": "mixed",
           "check_results": checks,
           "note": "inputs larger than L2; grid counts by Algorithm 2 (kappa0 = 20) before the timed region"}
    for p in plans:
        p.close()
    # the same batch on the plain FP64 path (same L-grids, samples and team size)
    fopts = dict(PATH_OPTIONS["fp64"])
    with ThreadPoolExecutor(16) as ex:
        plans = list(ex.map(lambda w: F.Plan(w.support, w.sizes, w.nodes, **fopts), ws))
    hs = [p.handle for p in plans]
    reps64 = F.fct_execute_batch(hs, xs, cs, team_blocks=tb)
    ms64 = statistics.mean(_timed(lambda: F.fct_execute_batch(hs, xs, cs, team_blocks=tb, report=False), 2,
                                  torch.empty(1, device="cuda")))
    out["fp64_path"] = {"value": sum_n / (ms64 / 1e3), "ms_per_launch": ms64,
                        "all_converged": all(r["status"] == 0 for r in reps64),
                        "max_iterations": max(r["iterations"] for r in reps64)}
    out["mixed_over_fp64"] = out["value"] / out["fp64_path"]["value"]
    for p in plans:
        p.close()
    return out


# ---------------------------------------------------------------------------
# serving leg: Poisson arrivals over shapes of D = 2..20, continuous batching
# ---------------------------------------------------------------------------
def serving_workloads(kappa0: float, probe_iterations: int = 200):
    """The serving plan shapes (one per D, |support| in [1e3, 1e5]) with the
    grid count picked by Algorithm 2 from a candidate L-grid of 10 D grids,
    probing from 3D grids on.  A shape whose candidates never reach kappa0
    takes the probed prefix with the least kappa x L (iterations x work per
    iteration)."""
    import workloads as W
    from paper_2309_14584_gb300 import lgrid
    from concurrent.futures import ThreadPoolExecutor

    def select(cand):
        t0 = time.perf_counter()
        r = lgrid.select_grids(cand.support, cand.sizes, cand.nodes, kappa0=kappa0, start=3 * cand.D,
                               step=max(1, cand.D // 2), probe_iterations=probe_iterations)
        L = r["L"]
        if L is None:
            L = min(r["probes"], key=lambda k: r["probes"][k] * k)
            r["kappa"] = r["probes"][L]
        return W.first_grids(cand, L), {"D": cand.D, "d": cand.d, "N": cand.N, "L": L, "kappa_est": r["kappa"],
                                        "probes": len(r["probes"]), "select_s": round(time.perf_counter() - t0, 3)}

    with ThreadPoolExecutor(8) as ex:   # plan building is host work; the library releases the GIL
        out = list(ex.map(select, W.serving_shapes(grids_per_dim=10)))
    return [o[0] for o in out], [o[1] for o in out]


def run_serving(args, F):
    import dataclasses
    import numpy as np
    import torch

    import workloads as W
    from paper_2309_14584_gb300.serving import ServingEngine, latency_summary

    rates = [float(x) for x in args.serving_rates.split(",") if x.strip()]
    if not rates:
        return None
    t0 = time.perf_counter()
    shapes, sel = serving_workloads(args.serving_kappa0)
    t_select = time.perf_counter() - t0
    team_tuning = []
    if args.serving_team_blocks <= 0:
        # blocks per team by measurement: a burst of every shape twice, per candidate
        for tb in (16, 38, 76):
            e = ServingEngine(shapes, hbm_budget_bytes=16e9, max_slots_per_shape=2, team_blocks=tb,
                              precision=F.FCT_MIXED, tol=1e-12, inner_tol=1e-4, max_iter=20000)
            xs = {}
            for s, w in enumerate(shapes):
                x = torch.empty(e.plans[s].M, dtype=torch.float64, device="cuda")
                e.plans[s].sample(W.FAMILY_GAUSSCOS, W.gausscos_params(w.D * 1000, w.D), x)
                xs[s] = x
            burst = [(0.0, s, s) for s in range(len(shapes))] * 2
            o = [torch.empty(e.plans[s].N, dtype=torch.float64, device="cuda") for _, s, _ in burst]
            e.run(burst[:len(shapes)], xs, o[:len(shapes)])          # warm-up
            t1 = time.perf_counter()
            e.run(burst, xs, o)
            team_tuning.append((tb, time.perf_counter() - t1))
            e.close()
            del xs, o
        team_blocks = min(team_tuning, key=lambda t: t[1])[0]
    else:
        team_blocks = args.serving_team_blocks
    eng = ServingEngine(shapes, hbm_budget_bytes=16e9, max_slots_per_shape=4, team_blocks=team_blocks,
                        precision=F.FCT_MIXED, tol=1e-12, inner_tol=1e-4, max_iter=20000)
    inputs, truth = {}, {}
    for s, w in enumerate(shapes):
        p = eng.plans[s]
        for v in range(SERVING_VARIANTS):
            x = torch.empty(p.M, dtype=torch.float64, device="cuda")
            p.sample(W.FAMILY_GAUSSCOS, W.gausscos_params(w.D * 1000 + v, w.D), x)
            inputs[(s, v)] = x
        c = W.poly_coefficients(w.D * 1000 + 999, w.support)
        x = torch.empty(p.M, dtype=torch.float64, device="cuda")
        p.sample(W.FAMILY_POLY, c, x)
        inputs[(s, "poly")] = x
        truth[s] = c
    torch.cuda.synchronize()
    # untimed warm-up: every shape once, all at t = 0
    warm = [(0.0, s, (s, 0)) for s in range(len(shapes))]
    eng.run(warm, inputs, [torch.empty(eng.plans[s].N, dtype=torch.float64, device="cuda") for _, s, _ in warm])
    out = []
    served = {}   # (shape, variant) -> coefficients served at the highest rate (results in the mix)
    for rate in rates:
        raw = W.serving_requests(5, args.serving_requests, rate, len(shapes), poly_fraction=0.05)
        reqs = [(t, s, (s, "poly") if poly else (s, ps % SERVING_VARIANTS)) for t, s, poly, ps in raw]
        outs = [torch.empty(eng.plans[s].N, dtype=torch.float64, device="cuda") for _, s, _ in reqs]
        res = eng.run(reqs, inputs, outs, timeout_s=300)
        summ = latency_summary(res, [eng.plans[s].N for _, s, _ in reqs])
        errs = [float(np.linalg.norm(o.cpu().numpy() - truth[s]) / np.linalg.norm(truth[s]))
                for (t, s, key), o in zip(reqs, outs) if key[1] == "poly"]
        summ.update(rate_req_s=rate, poly_requests=len(errs), poly_max_rel_err=max(errs) if errs else None,
                    max_iterations=max(r["report"]["iterations"] for r in res))
        out.append(summ)
        if rate == max(rates):
            for (t, s, key), o in zip(reqs, outs):
                if key[1] != "poly" and shapes[s].N <= SERVING_CHECK_MAX_N:
                    served.setdefault(key, o.cpu().numpy())
    eng.close()
    cold = run_serving_cold(args, F, shapes, inputs, team_blocks)
    checks = []
    for (s, v), c in sorted(served.items()):
        w = dataclasses.replace(shapes[s], params=W.gausscos_params(shapes[s].D * 1000 + v, shapes[s].D))
        checks.append((f"served:{w.name}_v{v}", w, c))
    return {"config": "Poisson arrivals over 19 shapes (D = 2..20, total degree d with |support| in [1e3, 1e5]), "
                      "Gaussian-cosine targets plus 5 % seeded polynomials (exact-recovery check), mixed path "
                      f"to 1e-12 normal residual; grid counts by Algorithm 2 with kappa0 = {args.serving_kappa0}; "
                      f"served Gaussian-cosine results of shapes with N <= {SERVING_CHECK_MAX_N} at the highest "
                      "rate are compared with the CPU oracle",
            "grid_selection_s": round(t_select, 2), "shapes": sel, "rates": out, "cold_plans": cold,
            "team_blocks": team_blocks, "team_blocks_tuning_s": [[t, round(x, 3)] for t, x in team_tuning],
            "check_results": checks}


def run_serving_cold(args, F, shapes, inputs, team_blocks, rate=25.0, n_req=60):
    """Plan-cache misses while serving: a fresh engine holds no plan; each
    shape's plan is built when its first request is admitted (grid counts as
    chosen by Algorithm 2 beforehand), while the serving launch runs on all
    teams but one (the free SMs run the plan builder's kernels).  Cold
    requests (their latency includes the plan build) are reported apart from
    the warm ones of the same run."""
    import numpy as np
    import workloads as W
    from paper_2309_14584_gb300.serving import ServingEngine
    eng = ServingEngine(shapes, hbm_budget_bytes=16e9, max_slots_per_shape=4, team_blocks=team_blocks,
                        teams=max(1, 304 // team_blocks - 1), lazy_plans=True, precision=F.FCT_MIXED,
                        tol=1e-12, inner_tol=1e-4, max_iter=20000)
    raw = W.serving_requests(9, n_req, rate, len(shapes), poly_fraction=0.0)
    reqs = [(t, s, (s, ps % SERVING_VARIANTS)) for t, s, _, ps in raw]
    outs = [torch_empty(shapes[s].N) for _, s, _ in reqs]
    res = eng.run(reqs, inputs, outs, timeout_s=300)
    builds = [1e3 * eng.plan_build_s[s] for s in sorted(eng.plan_build_s)]
    eng.close()
    cold = [1e3 * r["latency_s"] for r in res if r["cold"]]
    warm = [1e3 * r["latency_s"] for r in res if not r["cold"]]
    return {"requests": len(res), "rate_req_s": rate, "cold_requests": len(cold),
            "cold_p50_ms": float(np.percentile(cold, 50)) if cold else None,
            "cold_max_ms": max(cold) if cold else None,
            "warm_p50_ms": float(np.percentile(warm, 50)) if warm else None,
            "plan_build_ms_p50": float(np.percentile(builds, 50)) if builds else None,
            "plan_build_ms_max": max(builds) if builds else None,
            "all_converged": all(r["report"]["status"] == 0 for r in res),
            "note": "plans built on first request while the serving launch runs on all teams but one"}


def torch_empty(n):
    import torch
    return torch.empty(n, dtype=torch.float64, device="cuda")


# ---------------------------------------------------------------------------
# reference arm: the CPU oracle, as it stands, on the host cores
# ---------------------------------------------------------------------------
def run_reference(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return
    w = workload()
    # estimate one whole transform, then size each step so the run stays bounded
    probe = run_oracle(timing={"workload": "config_d10_rational", "budget_s": 0.0, "steps": 1})
    t_full = float(probe["times"][0])
    total_steps = args.steps + args.warmup
    fraction = min(1.0, REF_BUDGET_S / max(total_steps * t_full, 1e-9))
    res = run_oracle(timing={"workload": "config_d10_rational", "budget_s": 0.0, "steps": total_steps,
                             "fraction": fraction})
    times = res["times"][args.warmup:]
    credited = res["credited"][args.warmup:]
    value = float(credited.sum() / times.sum())
    host = cpu_description()
    line = {
        "impl": "reference",
        "metric": METRIC,
        "value": value,
        "unit": UNIT,
        "n_gpus": world,
        "steps": args.steps,
        "warmup": args.warmup,
        "ms_per_step": float(times.mean() * 1e3),
        "higher_is_better": True,
        "scaling": "weak",
        "vs_baseline": None,
        "dtype": "f64",
        "data": "synthetic",
        "config": workload_config(w),
        "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle",
                         "sample": f"each step = {fraction:.3f} of one transform (that share of the grids' "
                                   f"DCT-I and of the CGLS iterations), credited {fraction:.3f} x N coefficients",
                         "nproc": host["nproc"], "cpu_model": host["cpu_model"]},
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line))


def tc_profile_workload():
    """D=2, total degree 300 (N = 45451), 8 grids by Algorithm 1 with axes of
    150 to 301 points (M = 322576 samples), Gaussian-cosine target: a plan
    whose DCT runs on the tensor cores (the solve needs about 20 CG
    iterations, so the DCT is a large share of the transform)."""
    import workloads as W
    sup = W.total_degree_support(2, 300)
    sizes, nodes = W.l_grid(24, sup.shape[0], 2, 8, 150, 301)
    return W.Workload("D2_d300_gausscos_K8", 2, 300, sup, sizes, nodes, W.FAMILY_GAUSSCOS, W.gausscos_params(24, 2),
                      None, 1e-12, "mixed")


def sparse_profile_workload():
    """Sparse S^inf support at D = 100 (N = 2e4, 3 nonzero components per
    index, degree <= 9), 1000 grids, seeded polynomial target."""
    import workloads as W
    D, d, N = 100, 9, 20_000
    sup = W.sparse_infinity_support(13, D, d, N, 3)
    sizes, nodes = W.l_grid(300, N, D, 10 * D, 1, d + 1)
    c = W.poly_coefficients(10, sup)
    return W.Workload("sparse_D100_N2e4_K1000", D, d, sup, sizes, nodes, W.FAMILY_POLY, c, c, 1e-12, "mixed")


def sparse10_profile_workload():
    """Sparse S^inf support at D = 100 (N = 1e5, 10 nonzero components of degree
    <= 3 per index), 240 grids, seeded polynomial target: rows of every length
    from 1 to ~37k entries."""
    import workloads as W
    D, d, N, K = 100, 3, 100_000, 240
    sup = W.sparse_support_vectorised(3, D, d, N, 10)
    sizes, nodes = W.l_grid(500, N, D, K, 1, d + 1)
    c = W.poly_coefficients(10, sup)
    return W.Workload("sparse10_D100_N1e5_K240", D, d, sup, sizes, nodes, W.FAMILY_POLY, c, c, 1e-12, "mixed")


def run_profile(args):
    """`--warmup` + `--steps` executes of one case, nothing timed or printed
    but one status line: the command that ncu captures."""
    import torch
    import workloads as W
    import paper_2309_14584_gb300 as F
    from paper_2309_14584_gb300 import build as B
    B.build()
    torch.cuda.set_device(0)
    wname, path, popts = PROFILE_CASES[args.profile]
    w = getattr(W, wname)() if hasattr(W, wname) else globals()[wname]()
    plan = F.Plan(w.support, w.sizes, w.nodes, **dict(PATH_OPTIONS[path], **popts))
    x = torch.empty(plan.M, dtype=torch.float64, device="cuda")
    fam = w.family | (F.fct.FCT_SAMPLE_FOLDED if w.family == W.FAMILY_POLY else 0)
    plan.sample(fam, w.params, x)
    c = torch.empty(plan.N, dtype=torch.float64, device="cuda")
    rep = None
    for _ in range(args.warmup + args.steps):
        rep = plan.execute(x, c)
    torch.cuda.synchronize()
    print(json.dumps({"profile": args.profile, "workload": w.name, "N": plan.N, "M": plan.M,
                      "R": plan.info["R"], "K": plan.info["K"], "tensor_dct_grids": plan.info["tensor_dct_grids"],
                      "row_units": plan.info["row_units"], "wide_rows": plan.info["wide_rows"],
                      "coef_chunks": plan.info["coef_chunks"], "coef_split": plan.info["coef_split"],
                      "block_threads": plan.info["block_threads"], "grid_blocks": plan.info["grid_blocks"],
                      "report": rep}))
    plan.close()


def main():
    args = parse()
    if args.oracle_worker:
        oracle_worker(args.oracle_worker)
        return
    if args.profile:
        run_profile(args)
        return
    if args.impl == "reference":
        run_reference(args)
    else:
        run_gpu(args)


if __name__ == "__main__":
    main()
