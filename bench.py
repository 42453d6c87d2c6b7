#!/usr/bin/env python
"""Benchmark of the SVT hot path on GB300: one step = one complete matrix-completion solve.

Workload (default): 30000 x 30000, rank 10, |Omega| = 6 r (2n - r) = 3,599,400 sampled entries
(0.4 % of 9e8 unknowns), N(0,1) planted factors, tau = 5n, delta = 1.2/p, eps = 1e-4 -- the last
row of the paper's Table 1 -- with float64 values, sparse products, Lanczos basis and projected
SVD (the paper's arithmetic: Matlab double).  Steps cycle over the instances of seeds 0-4 (Table 1
averages five random instances); every instance counts, converged or not (k_max iterations).

A step runs the whole path through the C-ABI: svt_create (Omega storage: CSR, CSC, permutation),
svt_solve (kick with ||P_Omega M||_2, then Algorithm 1 until the relative residual on Omega is
<= 1e-4 or k_max iterations) and svt_destroy.  `value` is SVT iterations per second over the timed
steps (inputs resident in HBM); `e2e` is the same metric with the inputs copied from pinned host
memory and the factors of X copied back inside every step (one pass over the seeds).

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                    [--config NAME] [--precision fp64|fp32|bf16] [--seeds 0,1,2,3,4] [--k-max 1000]
    python bench.py --ncu-iters N ...   bounded run for a profiler: one create + kick + N
                                        iterations of the first seed, nothing timed (shrink
                                        decided on the host: ncu skips conditional graphs)

Under torchrun each rank solves its own problems (seed + 1000 rank): weak scaling, no data-path
collective; the timing is the maximum over ranks.
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from svt_inputs import CONFIGS, config_problem  # noqa: E402

METRIC = "SVT iters/s to 1e-4 rel. residual (time-to-1e-4 per solve)"
PEAKS_FILE = os.path.join(ROOT, "MEASURED_PEAKS.json")
TRAFFIC_FILE = os.path.join(ROOT, "profiles", "traffic.json")
FALLBACK_HBM_GBS = 6800.0


def _peaks():
    try:
        with open(PEAKS_FILE) as f:
            p = json.load(f)
        return float(p["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM_GBS, "fallback"


# Arithmetic peaks derived from GB300's unit counts at the maximum SM clock (2070 MHz, 152 SMs):
# float64 2 FMA / clock / SM (1.26 TFLOP/s, the nominal 1.25), float32 128 FMA / clock / SM.
SM_COUNT, SM_MAX_HZ = 152, 2.070e9
PEAK_FP64_TFLOPS = SM_COUNT * 2 * 2 * SM_MAX_HZ / 1e12
PEAK_FP32_TFLOPS = SM_COUNT * 128 * 2 * SM_MAX_HZ / 1e12


def _kernel_source_sha():
    h = hashlib.sha256()
    csrc = os.path.join(ROOT, "paper_0810_3286_gb300", "csrc")
    for name in sorted(os.listdir(csrc)):
        with open(os.path.join(csrc, name), "rb") as f:
            h.update(f.read())
    return h.hexdigest()[:16]


def _traffic_for(kernel_class, precision):
    """DRAM bytes per launch (dram__bytes_read.sum + dram__bytes_write.sum, averaged over the captured
    launches of the class) from the committed ncu summary of this precision's profiling run, if it
    was taken on the current kernel source; None otherwise."""
    try:
        with open(TRAFFIC_FILE) as f:
            t = json.load(f)
    except Exception:
        return None
    if t.get("csrc_sha") != _kernel_source_sha():
        return None
    entry = t.get("classes_" + precision, {}).get(kernel_class)
    return None if entry is None else float(entry)


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled every 200 ms during the timed region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, device_index):
        self.device_index = device_index
        self.proc = None
        log_dir = os.environ.get("SVT_BENCH_LOG_DIR", os.path.join(ROOT, "bench_logs"))
        self.path = os.path.join(log_dir, "clocks_rank%d.csv" % device_index)

    def start(self):
        try:
            os.makedirs(os.path.dirname(self.path), exist_ok=True)
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "--query-gpu=" + self.FIELDS, "--format=csv,noheader,nounits",
                                          "-lms", "200", "-i", str(self.device_index)], stdout=self.f,
                                         stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.f.close()
        sm, smax, reasons = [], [], set()
        names = ["active", "hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        with open(self.path) as f:
            for line in f:
                parts = [x.strip() for x in line.split(",")]
                if len(parts) < 9:
                    continue
                try:
                    sm.append(float(parts[1]))
                    smax.append(float(parts[2]))
                except ValueError:
                    continue
                for nm, v in zip(names[1:], parts[5:9]):
                    if v.lower() == "active":
                        reasons.add(nm)
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": float(np.median(sm)), "sm_max_mhz": float(max(smax)), "reasons": sorted(reasons),
                "samples": len(sm)}


def _dist():
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch
        import torch.distributed as dist
        backend = "nccl" if torch.cuda.is_available() else "gloo"
        dist.init_process_group(backend=backend)
        return world, rank, local, dist
    return world, rank, local, None


def _max_over_ranks(dist, value, device):
    if dist is None:
        return value
    import torch
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def _sum_over_ranks(dist, value, device):
    if dist is None:
        return value
    import torch
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.SUM)
    return float(t.item())


def _barrier(dist):
    if dist is not None:
        dist.barrier()


def _cpu_model():
    """CPU model and core count of the host (lscpu where available)."""
    model = None
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.split(":")[0].strip() in ("Model name", "Model"):
                v = line.split(":", 1)[1].strip()
                if v and not v.isdigit():
                    model = v
                    break
    except Exception:
        pass
    if model is None:
        import platform
        model = platform.processor() or platform.machine()
    return model, os.cpu_count() or 1


def _oracle_iterations(config_name, seed, first, count, threads):
    """The float64 sparse-tier oracle (oracle/svt_sparse.py) as it stands, on the host cores: Algorithm 1
    from the kick (||P_Omega M||_2 by the oracle's partial SVD, k0 of eq. (5.3)) through iteration
    first + count - 1.  Returns the seconds of iterations first .. first + count - 1 (timed between the
    per-iterate callbacks; the kick and earlier iterations are untimed set-up).  `threads` caps the
    BLAS threads of the oracle's dense steps (its sparse products are single-threaded scipy)."""
    code = r"""
import json, sys, time
sys.path.insert(0, %r)
from oracle import svt_sparse
from svt_inputs import config_problem
p = config_problem(%r, %d)
stamps = {}
def cb(rec):
    stamps[rec.k] = time.perf_counter()
first, count = %d, %d
svt_sparse.svt(p.n1, p.n2, p.rows, p.cols, p.vals, p.tau_default(), p.delta_default(), k_max=first + count - 1,
               keep_trace=False, on_iter=cb)
ks = sorted(stamps)
t0 = stamps[first - 1]
t1 = stamps[ks[-1]]
print(json.dumps({"seconds": t1 - t0, "iters": ks[-1] - (first - 1)}))
""" % (ROOT, config_name, seed, first, count)
    env = dict(os.environ)
    for v in ("OPENBLAS_NUM_THREADS", "OMP_NUM_THREADS", "MKL_NUM_THREADS"):
        env[v] = str(threads)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, env=env)
    if r.returncode != 0:
        raise RuntimeError("oracle run failed:\n" + r.stderr[-2000:])
    out = json.loads(r.stdout.strip().splitlines()[-1])
    return out["seconds"], out["iters"]


def cpu_baseline(config_name, seed, single_thread=False):
    """The float64 sparse-tier oracle on the host cores, on a bounded sample of the workload: SVT
    iteration 2 of the instance (kick and iteration 1 untimed), with the BLAS threads at the core
    count (and again at one thread with single_thread: the oracle's sparse products are
    single-threaded scipy, so the two rates are within a few per cent)."""
    model, cores = _cpu_model()
    c = CONFIGS[config_name]
    t_all, n_all = _oracle_iterations(config_name, seed, 2, 1, cores)
    line = {"value": n_all / t_all, "unit": "iters/s", "cores": cores, "kind": "oracle",
            "sample": "SVT iteration 2 of the %dx%d rank-%d instance of seed %d (kick and iteration 1 untimed), "
                      "float64 sparse-tier oracle (scipy sparse products, block subspace iteration, Jacobi SVD), "
                      "BLAS threads = %d, %.1f s timed" % (c["n1"], c["n2"], c["r"], seed, cores, t_all),
            "cpu_model": model}
    if single_thread:
        t_one, n_one = _oracle_iterations(config_name, seed, 2, 1, 1)
        line["single_thread"] = {"value": n_one / t_one, "unit": "iters/s", "cores": 1, "seconds": t_one}
    return line


def run_reference(args):
    """The reference arm: the float64 oracle as it stands on the host cores.  Its kick and W warm-up
    iterations are untimed; then `steps` SVT iterations are timed.  Under torchrun only rank 0 runs
    it; the other ranks exit without work (no process group is needed)."""
    if int(os.environ.get("RANK", "0")) != 0:
        return 0
    c = CONFIGS[args.config]
    seed = args.seed_list[0]
    model, cores = _cpu_model()
    steps = max(1, args.steps)
    dt, n = _oracle_iterations(args.config, seed, 2 + args.warmup, steps, cores)
    v = n / dt
    p = config_problem(args.config, seed)
    sample = ("SVT iterations %d..%d of the %dx%d rank-%d instance of seed %d (kick and earlier iterations "
              "untimed), float64 sparse-tier oracle, BLAS threads = %d, %.1f s timed"
              % (2 + args.warmup, 1 + args.warmup + n, c["n1"], c["n2"], c["r"], seed, cores, dt))
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "iters/s", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000.0 * dt / n,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": _config_dict(args, p.nnz, 1),
            "cpu_baseline": {"value": v, "unit": "iters/s", "cores": cores, "kind": "oracle", "sample": sample,
                             "cpu_model": model},
            "e2e": {"value": v, "unit": "iters/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


def _config_dict(args, nnz, world):
    c = CONFIGS[args.config]
    return {"workload": "%s: %dx%d rank %d, |Omega|=%d (6 r(2n-r)), tau=5n, delta=1.2/p, eps=1e-4"
                        % (args.config, c["n1"], c["n2"], c["r"], nnz),
            "precision": {"fp64": "float64 values and sparse products, float64 Lanczos basis and projected SVD",
                          "fp32": "float32 values and sparse products (float32 accumulation), float64 Lanczos basis "
                                  "and projected SVD",
                          "bf16": "bfloat16 values in the sparse products while the residual is above 1e-2, then "
                                  "float32 (float32 accumulation), float64 Lanczos basis and projected SVD"}[args.precision],
            "step": "svt_create (Omega storage) + svt_solve (kick + iterations to 1e-4, at most k_max) + "
                    "svt_destroy, one problem instance per step",
            "seeds": args.seed_list, "k_max": args.k_max,
            "l2": "inputs larger than L2 and a 256 MB buffer written between steps (flush)",
            "parallelism": "replicas%d" % world}


def run_ncu(args):
    """Bounded run for a profiler: create, kick and `ncu_iters` SVT iterations of the first seed."""
    import torch
    from paper_0810_3286_gb300 import Solver, build
    build.build()
    torch.cuda.set_device(0)
    p = config_problem(args.config, seed=args.seed_list[0])
    # ncu does not profile kernel nodes of graphs that hold conditional nodes, so the bounded run
    # decides the shrink on the host (the same kernels with the same launch shapes, one graph per
    # Lanczos cycle)
    with Solver(p.n1, p.n2, torch.from_numpy(p.rows).cuda(), torch.from_numpy(p.cols).cuda(),
                torch.from_numpy(p.vals).cuda(), precision=args.precision, device_loop=False) as s:
        s.configure(p.tau_default(), p.delta_default(), 1e-4, 27)
        k = 0
        for k in range(args.ncu_iters):
            if s.step()["stopped"]:
                break
        torch.cuda.synchronize()
        print(json.dumps({"ncu_run": args.config, "precision": args.precision, "seed": args.seed_list[0],
                          "iterations": k + 1, "counters": s.counters()}))
    return 0


def run_ours(args):
    import torch
    world, rank, local, dist = _dist()
    torch.cuda.set_device(local)
    device = torch.device("cuda", local)
    from paper_0810_3286_gb300 import Solver, build
    build.build()
    from paper_0810_3286_gb300 import _abi
    stream = torch.cuda.current_stream()

    seeds = [sd + 1000 * rank for sd in args.seed_list]
    probs = [config_problem(args.config, seed=sd) for sd in seeds]
    dev_in = [(torch.from_numpy(p.rows).to(device), torch.from_numpy(p.cols).to(device),
               torch.from_numpy(p.vals).to(device)) for p in probs]
    host_in = [(torch.from_numpy(p.rows).pin_memory(), torch.from_numpy(p.cols).pin_memory(),
                torch.from_numpy(p.vals).pin_memory()) for p in probs]
    l2_flush = torch.empty(64 * 1024 * 1024, dtype=torch.float32, device=device)  # 256 MB > 129 MB L2
    p0 = probs[0]
    cap = 27

    def step_device(i, profile_classes=(), k_max=None):
        p = probs[i]
        rows_d, cols_d, vals_d = dev_in[i]
        s = Solver(p.n1, p.n2, rows_d, cols_d, vals_d, precision=args.precision, stream=stream,
                   k_max=k_max or args.k_max)
        if profile_classes:
            s.set_profile(profile_classes)
        res = s.solve(p.tau_default(), p.delta_default(), 1e-4, cap, raise_on_nonconvergence=False)
        prof = s.profile() if profile_classes else None
        launches = s.kernel_launches()
        step_device.counters = s.counters()
        s.close()
        return res, launches, prof

    U_h = torch.empty((max(p.n1 for p in probs), cap), dtype=torch.float64).pin_memory()
    d_h = torch.empty(cap, dtype=torch.float64).pin_memory()
    V_h = torch.empty((max(p.n2 for p in probs), cap), dtype=torch.float64).pin_memory()

    def step_e2e(i):
        p = probs[i]
        rows_h, cols_h, vals_h = host_in[i]
        s = Solver(p.n1, p.n2, rows_h.numpy(), cols_h.numpy(), vals_h.numpy(), precision=args.precision,
                   stream=stream, k_max=args.k_max)
        res = s.solve(p.tau_default(), p.delta_default(), 1e-4, cap, raise_on_nonconvergence=False)
        r = res["rank"]
        st = s._L.svt_get_factors(s._ctx, U_h.data_ptr(), d_h.data_ptr(), V_h.data_ptr(), cap)
        assert st == 0
        s.close()
        return res, r

    nseed = len(probs)
    # --- warm-up: the same create / solve / destroy, capped at 30 iterations ---
    for k in range(args.warmup):
        step_device(k % nseed, k_max=30)
    # --- per-class profile of one untimed solve (first 150 iterations of the first instance) ---
    _, _, prof_all = step_device(0, tuple(_abi.PROF_CLASSES), k_max=min(args.k_max, 150))
    shares = {k: v[1] for k, v in prof_all.items()}
    tot = sum(shares.values()) or 1.0
    dominant_all = max(shares, key=lambda k: shares[k])

    # --- timed region: K device-resident steps, nothing instrumented ---
    clocks = ClockSampler(torch.cuda.current_device())
    _barrier(dist)
    torch.cuda.synchronize()
    clocks.start()
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    iters = 0
    launches = 0
    results = []
    counters = []
    t_wall0 = time.perf_counter()
    for k in range(args.steps):
        l2_flush.zero_()
        ev[k][0].record(stream)
        res, nl, _ = step_device(k % nseed)
        ev[k][1].record(stream)
        iters += res["iterations"]
        launches += nl
        results.append(res)
        counters.append(dict(step_device.counters))
    torch.cuda.synchronize()
    t_wall = time.perf_counter() - t_wall0
    _barrier(dist)
    clk = clocks.stop()
    step_ms = [a.elapsed_time(b) for a, b in ev]
    total_s = sum(step_ms) / 1000.0
    total_s_max = _max_over_ranks(dist, total_s, device)
    iters_all = _sum_over_ranks(dist, float(iters), device)
    value = iters_all / total_s_max

    # --- roofline pass: one solve per instance (at most 150 iterations each) with CUDA events (on the
    # library's stream, recorded by the captured graphs) around every launch of every kernel class ---
    prof_timed = {}
    for i in range(nseed):
        l2_flush.zero_()
        _, _, prof = step_device(i, tuple(_abi.PROF_CLASSES), k_max=min(args.k_max, 150))
        for c, (n, ms, by, fl) in prof.items():
            a = prof_timed.setdefault(c, [0, 0.0, 0.0, 0.0])
            a[0] += n; a[1] += ms; a[2] += by; a[3] += fl
    torch.cuda.synchronize()

    # --- end to end through the C-ABI with host buffers: one pass over the instances ---
    step_e2e(0)
    _barrier(dist)
    torch.cuda.synchronize()
    e2e_iters, e2e_bi, e2e_bo = 0, 0, 0
    e2e_ev = []
    for k in range(nseed):
        l2_flush.zero_()
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record(stream)
        res, r = step_e2e(k)
        b.record(stream)
        e2e_ev.append((a, b))
        e2e_iters += res["iterations"]
        e2e_bi += probs[k].nnz * (4 + 4 + 8)
        e2e_bo += 8 * (probs[k].n1 + probs[k].n2 + 1) * r
    torch.cuda.synchronize()
    e2e_s = sum(a.elapsed_time(b) for a, b in e2e_ev) / 1000.0
    e2e_s = _max_over_ranks(dist, e2e_s, device)
    e2e_iters = _sum_over_ranks(dist, float(e2e_iters), device)
    _barrier(dist)

    if rank != 0:
        if dist is not None:
            dist.destroy_process_group()
        return 0

    peak, peak_kind = _peaks()

    def _sum(classes, i):
        return sum(prof_timed.get(c, [0, 0.0, 0.0, 0.0])[i] for c in classes)

    def _roof(classes, name):
        n_l, ms_l, by_l = _sum(classes, 0), _sum(classes, 1), _sum(classes, 2)
        achieved = (by_l / 1e9) / (ms_l / 1e3) if ms_l > 0 else None
        return {"bound": "hbm", "kernel": name, "achieved": achieved, "peak": peak, "unit": "GB/s",
                "frac": (achieved / peak) if achieved else None, "peak_kind": "%s copy bandwidth" % peak_kind,
                "traffic": _traffic_for(classes[0], args.precision), "launches_timed": n_l,
                "avg_launch_us": 1000.0 * ms_l / n_l if n_l else None,
                "algorithmic_bytes_per_launch": by_l / n_l if n_l else None}

    def _roof_alu(cls, name, flops_total, peak_tflops, kind):
        classes = cls if isinstance(cls, tuple) else (cls,)
        cls = classes[0]
        n_l, ms_l = _sum(classes, 0), _sum(classes, 1)
        achieved = (flops_total / 1e12) / (ms_l / 1e3) if ms_l > 0 else None
        return {"bound": "alu", "kernel": name, "achieved": achieved, "peak": peak_tflops, "unit": "TFLOP/s",
                "frac": (achieved / peak_tflops) if achieved else None,
                "peak_kind": "%s peak derived from unit counts x maximum SM clock" % kind,
                "traffic": _traffic_for(cls, args.precision), "launches_timed": n_l,
                "avg_launch_us": 1000.0 * ms_l / n_l if n_l else None,
                "algorithmic_flops_per_launch": flops_total / n_l if n_l else None}

    # float64 values: the sparse products issue b float64 FMAs per sampled entry and are bound by
    # the float64 pipe, so their roofline is the float64 peak; float32 values: the
    # streamed bytes against the copy bandwidth
    if args.precision == "fp64":
        roof_spmm = lambda: _roof_alu(("spmm", "spmm_t"), "k_spmm (Y V and Y^T U, float64)",
                                      _sum(("spmm", "spmm_t"), 3), PEAK_FP64_TFLOPS, "float64")
    else:
        roof_spmm = lambda: _roof(("spmm", "spmm_t"), "k_spmm (Y V and Y^T U)")
    rooflines = {
        "orth": lambda: dict(_roof_alu("orth", "k_orth_coop (block CGS2 + Cholesky QR, float64 accuracy)",
                                       _sum(("orth",), 3), PEAK_FP64_TFLOPS, "float64"),
                             note="most of the operations run as float16 digit products on the tensor cores: frac "
                                  "compares with the float64 pipe and is not its utilisation"),
        "spmm": roof_spmm,
        "spmm_t": roof_spmm,
        "sddmm_update": lambda: _roof(("sddmm_update",), "k_sddmm_update"),
    }
    timed_shares = {c: v[1] for c, v in prof_timed.items()}
    dominant = max(timed_shares, key=lambda c: timed_shares[c]) if timed_shares else "spmm"
    roofline = rooflines.get(dominant, rooflines["orth"])()
    roofline["time_share"] = timed_shares.get(dominant, 0.0) / (sum(timed_shares.values()) or 1.0)
    cpu = (cpu_baseline(args.config, args.seed_list[0], single_thread=args.cpu_single_thread)
           if not args.no_cpu_baseline else None)
    conv = [r for r in results if r["converged"]]
    per_seed = {}
    for k, r in enumerate(results):
        sd = seeds[k % nseed]
        e = per_seed.setdefault(str(sd), {"iterations": r["iterations"], "converged": bool(r["converged"]),
                                          "ms": [], "rank": r["rank"], "residual": r["residual"]})
        e["ms"].append(step_ms[k])
    for e in per_seed.values():
        e["ms"] = float(np.median(e["ms"]))
    cnt = {k: float(np.mean([c[k] for c in counters])) for k in counters[0]} if counters else {}
    line = {
        "metric": METRIC, "value": value, "unit": "iters/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": 1000.0 * total_s_max / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None,
        "dtype": {"fp64": "f64", "fp32": "f32", "bf16": "bf16"}[args.precision], "data": "synthetic",
        "config": _config_dict(args, p0.nnz, world),
        "time_to_1e-4_ms": (float(np.mean([step_ms[k] for k, r in enumerate(results) if r["converged"]]))
                            if conv else None),
        "converged_steps": len(conv), "per_seed": per_seed,
        "iterations_per_solve": float(np.mean([r["iterations"] for r in results])),
        "k0": results[0]["k0"], "wall_s": t_wall,
        "clocks": clk,
        "e2e": {"value": e2e_iters / e2e_s, "unit": "iters/s", "h2d_bytes_per_step": int(e2e_bi / nseed),
                "d2h_bytes_per_step": int(e2e_bo / nseed)},
        "gpu_launches": int(launches),
        "roofline": roofline,
        "roofline_spmm": roof_spmm(),
        "roofline_spmm_hbm": _roof(("spmm", "spmm_t"), "k_spmm (Y V and Y^T U)"),
        "roofline_update": _roof(("sddmm_update",), "k_sddmm_update"),
        "kernel_time_shares": {k: round(v / tot, 4) for k, v in shares.items()},
        "dominant_kernel_class": dominant_all,
        "solver_counters_per_solve": cnt,
        "cpu_baseline": cpu,
    }
    print(json.dumps(line))
    if dist is not None:
        dist.destroy_process_group()
    return 0


def main():
    ap = argparse.ArgumentParser(description=__doc__, formatter_class=argparse.RawDescriptionHelpFormatter)
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--config", default="large_30000", choices=sorted(CONFIGS))
    ap.add_argument("--precision", default="fp64", choices=["fp32", "fp64", "bf16"])
    ap.add_argument("--seeds", default="0,1,2,3,4",
                    help="problem instances the steps cycle over (rank k solves seed + 1000 k)")
    ap.add_argument("--k-max", type=int, default=1000, help="SVT iteration cap per solve")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-single-thread", action="store_true",
                    help="also time the CPU baseline with one BLAS thread")
    ap.add_argument("--ncu-iters", type=int, default=0,
                    help="bounded run for a profiler: create + kick + this many iterations, nothing timed")
    args = ap.parse_args()
    args.seed_list = [int(x) for x in args.seeds.split(",") if x.strip()]
    if not args.seed_list:
        ap.error("--seeds is empty")
    if args.ncu_iters > 0:
        return run_ncu(args)
    if args.warmup < 3 and args.impl == "ours":
        ap.error("--warmup must be >= 3")
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
