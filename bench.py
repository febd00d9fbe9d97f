#!/usr/bin/env python
"""Benchmark: l1-Cox proximal-gradient iterations/s on one GB300.

Workload (default): the paper-scale genotype problem -- n = 400,000 subjects,
p = 500,000 SNPs (2-bit packed, MAF ~ U(0.01, 0.5)), 500 causal SNPs, integer
days 1..5000 with ties, ~5% events, 16 penalties log-spaced from lambda_max to
0.01 lambda_max solved together.  A step is one proximal-gradient iteration
for all 16 penalties: X_c B, Breslow risk-set scans, X_c^T V, soft threshold.

The JSON line carries the device-timed throughput (inputs resident in HBM),
the end-to-end throughput through the C ABI with host buffers, the roofline
of the dominant kernel (the tensor-core genotype product), the plain FP32
GEMV path on the same resident data, and the FP64 oracle timed on a bounded
sample on the host cores.  ``--impl reference`` times only that oracle.
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

# the metric's published name; the operand form measured here is in the "precision" key
METRIC = "l1-Cox prox-grad iters/s & HBM GB/s: batched-lambda split-BF16 vs plain FP32"
UNIT = "iter/s"


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="geno_400k_500k_k16",
                    help="synthetic workload recipe (synth.WORKLOADS); --n/--p/--k rescale it")
    ap.add_argument("--n", type=int, default=None)
    ap.add_argument("--p", type=int, default=None)
    ap.add_argument("--k", type=int, default=None)
    ap.add_argument("--precision", default="split_e2m1", choices=["split_e4m3", "split_e2m1"],
                    help="operand form of the tensor-core products: e2m1 (kind::mxf4, eight limbs) or e4m3 "
                         "(kind::f8f6f4, four limbs)")
    ap.add_argument("--tile-m", type=int, default=0)
    ap.add_argument("--stages", type=int, default=0)
    ap.add_argument("--chunks", type=int, default=0)
    ap.add_argument("--window", type=int, default=0,
                    help="K chunks per TMEM accumulation window (0: the library default, 256)")
    ap.add_argument("--issue", type=int, default=0,
                    help="MMA issue mode of the products: 1 one issuer per row tile, 2 two on alternate stages")
    ap.add_argument("--no-autotune", action="store_true",
                    help="skip cox_autotune (the pipeline shapes then come from the built-in default)")
    ap.add_argument("--gemv-steps", type=int, default=2)
    ap.add_argument("--e2e-steps", type=int, default=5)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-gemv", action="store_true")
    ap.add_argument("--cpu-sample-cols", type=int, default=1000)
    ap.add_argument("--cpu-sample-steps", type=int, default=3)
    ap.add_argument("--path-iters", type=int, default=1000,
                    help="iteration cap of the timed cox_path_fit run (0: skip it)")
    ap.add_argument("--path-tol", type=float, default=1e-6)
    ap.add_argument("--nmf-iters", type=int, default=200,
                    help="timed iterations per NMF algorithm (Section 5.1, X 10,000 x 10,000); 0 skips it")
    ap.add_argument("--nmf-m", type=int, default=10_000)
    ap.add_argument("--nmf-n", type=int, default=10_000)
    ap.add_argument("--nmf-r", type=int, default=20)
    ap.add_argument("--nmf-only", action="store_true", help="run and print only the NMF object")
    ap.add_argument("--active-steps", type=int, default=5,
                    help="iterations timed with and without the active-set X B after the path fit (0: skip)")
    return ap.parse_args()


def recipe(args):
    import synth
    if args.workload not in synth.WORKLOADS:
        raise SystemExit(f"unknown workload {args.workload!r}; one of {sorted(synth.WORKLOADS)}")
    r = synth.WORKLOADS[args.workload]
    if args.n or args.p or args.k:
        r = r.scaled(n=args.n, p=args.p, k=args.k)
    return r


def workload_name(r) -> str:
    if r.kind != "geno":
        return (f"{r.name}: n={r.n} subjects x p={r.p} N(0,1) predictors, {r.n_causal} causal, "
                f"{r.cens_frac:.0%} censored, no ties, k={r.k} at {r.lam_hi} lambda_max")
    return (f"{r.name}: n={r.n} subjects x p={r.p} SNPs 2-bit packed, MAF~U({r.maf_lo},{r.maf_hi}), "
            f"{r.n_causal} causal, days 1..{r.dmax} (ties), {r.event_frac:.0%} events, k={r.k} lambdas "
            f"log-spaced lambda_max..{r.lam_lo} lambda_max")


def measured_peak_hbm():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    try:
        with open(path) as fh:
            d = json.load(fh)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


def gemm_traffic(k: int, n: int, p: int, precision: str):
    """DRAM bytes per launch of the tensor-core product from the committed ncu
    summary of its operand form, scaled by n*p codes; None when the kernel
    source changed since."""
    import hashlib
    form = "e2m1" if precision == "split_e2m1" else "e4m3"
    path = os.path.join(ROOT, "profiles", f"k_packed_gemm_{form}_traffic_n65536_p65536_k16.txt")
    src = os.path.join(ROOT, "paper_2010_16114_gb300", "csrc", "gemm_kernel.cuh")
    try:
        kv = {}
        with open(path) as fh:
            for line in fh:
                if ":" in line:
                    a, b = line.split(":", 1)
                    kv[a.strip()] = b.strip()
        with open(src, "rb") as fh:
            sha = hashlib.sha256(fh.read()).hexdigest()
        if kv.get("source_sha256") != sha or int(kv.get("k", -1)) != k:
            return None
        return float(kv["dram_bytes_per_code"]) * n * p
    except Exception:
        return None


def nmf_traffic(m: int, n: int, r: int):
    """DRAM bytes per launch of the NMF product from the committed ncu summary
    (taken at this workload's full size); None for another workload or when the
    kernel source changed since."""
    import hashlib
    path = os.path.join(ROOT, "profiles", "k_nmf_gemm_traffic_m10000_n10000_r20.txt")
    src = os.path.join(ROOT, "paper_2010_16114_gb300", "csrc", "nmf_gemm.cuh")
    try:
        kv = {}
        with open(path) as fh:
            for line in fh:
                if ":" in line:
                    a, b = line.split(":", 1)
                    kv[a.strip()] = b.strip()
        with open(src, "rb") as fh:
            sha = hashlib.sha256(fh.read()).hexdigest()
        if kv.get("source_sha256") != sha or (m, n, r) != (int(kv["m"]), int(kv["n"]), int(kv["r"])):
            return None
        return float(kv["dram_bytes_per_launch"])
    except Exception:
        return None


# ------------------------------------------------------------------ distributed plumbing
def dist_init(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        backend = "nccl" if args.impl == "ours" else "gloo"
        dist.init_process_group(backend=backend)
    return rank, world


def barrier(world):
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(x: float, world: int) -> float:
    if world == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device="cuda" if dist.get_backend() == "nccl" else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


# ------------------------------------------------------------------ clocks
class Clocks:
    """nvidia-smi samples every 200 ms while the timed region runs."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, dev: int):
        self.dev = dev
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-lms", "200", "-i", str(self.dev)], stdout=subprocess.PIPE,
                                         stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.25)
        self.proc.terminate()
        out, _ = self.proc.communicate(timeout=10)
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.strip().splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                smax.append(float(f[2]))
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


# ------------------------------------------------------------------ CPU oracle baseline
class OracleSample:
    """The FP64 oracle, as it stands, on a bounded sample of the workload: all n
    subjects, the first `cols` SNP columns, one penalty.  A step is one ISTA
    iteration of the oracle (Section 5.3): eta, the risk-set sums, the
    gradient, the soft threshold.  With one thread it is oracle.ista itself;
    with more, the oracle's own eta and gradient routines run concurrently on
    column blocks (each column's gradient is the oracle's; eta adds the
    blocks' partial sums), on the host's cores."""

    def __init__(self, r, cols: int):
        import oracle
        import synth
        oracle.build()
        self.oracle = oracle
        self.r = r
        self.w = synth.Workload(r)
        self.cols = min(cols, r.p)
        idx = np.arange(self.cols)
        if r.kind == "geno":
            X = self.w.cols_u8(idx, threads=os.cpu_count() or 1).T
        else:
            X = self.w.cols(idx)
        self.X = np.asfortranarray(X, dtype=np.float64)  # n x cols, column-major
        self.mu = self.X.mean(axis=0)

    def time_step(self, cols: int, threads: int, steps: int) -> float:
        """Median seconds of one oracle iteration on the first `cols` columns."""
        from concurrent.futures import ThreadPoolExecutor
        o, w = self.oracle, self.w
        X, mu = self.X[:, :cols], self.mu[:cols]
        sigma, lam = 1e-3, 0.0
        beta = np.zeros(cols)
        blocks = [b for b in np.array_split(np.arange(cols), threads) if len(b)]
        Xb = [np.asfortranarray(X[:, b]) for b in blocks]
        times = []
        with ThreadPoolExecutor(max(1, threads)) as ex:
            for _ in range(steps):
                t0 = time.perf_counter()
                if threads == 1:
                    beta, _, _ = o.ista(X, mu, w.y, w.delta, sigma, lam, 1, beta)
                else:
                    parts = list(ex.map(lambda q: o.eta(Xb[q], mu[blocks[q]], beta[blocks[q]]), range(len(blocks))))
                    eta = np.sum(parts, axis=0)
                    _, u, _ = o.risk(w.y, w.delta, eta)
                    gs = list(ex.map(lambda q: o.grad(Xb[q], mu[blocks[q]], w.delta, u), range(len(blocks))))
                    beta = o.prox(beta, np.concatenate(gs), sigma, lam)
                times.append(time.perf_counter() - t0)
        return float(np.median(times))

    def baseline(self, steps: int):
        """cpu_baseline object: the threaded oracle on all host cores, the
        1-thread figure beside it.  A step costs a fixed part per penalty (the
        risk-set sums over n subjects, their sort) plus a part per column (eta
        and the gradient), so one full iteration is extrapolated from the step
        times at two sample sizes, t(c) = a + b c, as k (a + b p)."""
        r = self.r
        cores = os.cpu_count() or 1
        half = max(1, self.cols // 2)
        t_all = self.time_step(self.cols, cores, steps)
        t_half = self.time_step(half, cores, steps)
        t_one = self.time_step(self.cols, 1, max(1, steps // 2))
        t_one_half = self.time_step(half, 1, max(1, steps // 2))

        def full(t_c, t_h):
            b = max((t_c - t_h) / (self.cols - half), 1e-12) if self.cols > half else t_c / self.cols
            a = max(t_c - b * self.cols, 0.0)
            return r.k * (a + b * r.p), a, b

        T, a, b = full(t_all, t_half)
        T1, a1, b1 = full(t_one, t_one_half)
        return {
            "value": 1.0 / T, "unit": UNIT, "cores": cores, "kind": "oracle",
            "sample": f"one FP64 oracle iteration (eta, risk-set sums, gradient, soft threshold) on all {r.n} "
                      f"subjects x the first {self.cols} and {half} SNP columns, one penalty, oracle routines on "
                      f"{cores} threads over column blocks, median of {steps}; a full iteration = {r.k} penalties x "
                      f"(a + b p) from the two step times",
            "step_s": {str(self.cols): t_all, str(half): t_half},
            "model_s": {"a_per_penalty": a, "b_per_column": b},
            "one_thread": {"value": 1.0 / T1, "unit": UNIT, "cores": 1,
                           "sample": f"oracle.ista itself on the same samples, median of {max(1, steps // 2)}",
                           "step_s": {str(self.cols): t_one, str(half): t_one_half},
                           "model_s": {"a_per_penalty": a1, "b_per_column": b1}},
        }


def run_reference(args, rank, world):
    if rank != 0:
        return 0
    r = recipe(args)
    smp = OracleSample(r, args.cpu_sample_cols)
    if args.warmup > 0:
        smp.time_step(min(smp.cols, 50), os.cpu_count() or 1, 1)
    cpu = smp.baseline(max(1, args.steps))
    value = cpu["value"]
    line = {
        "impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 / value, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": workload_name(r), "n": r.n, "p": r.p, "k": r.k},
        "cpu_baseline": cpu,
        "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
    }
    print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------------ our arm
NMF_PAPER_1GPU_S = {20: {"mult": 62, "apg": 61}, 40: {"mult": 72, "apg": 80}, 60: {"mult": 83, "apg": 85}}


def run_nmf(args, stream, cpu_baseline: bool = False):
    """Section 5.1 NMF on one GPU: X m x n (grid k / 256, exact in bf16), rank r,
    both algorithms; device-resident iterations timed with CUDA events, the two
    tensor-core products timed per launch for the roofline, and an end-to-end
    run from host factors to host factors."""
    import torch

    import synth
    from paper_2010_16114_gb300.nmf import NMF

    m, n, r = args.nmf_m, args.nmf_n, args.nmf_r
    X, V0, W0 = synth.nmf_inputs(m, n, r)
    h = NMF(X, r)
    info = h.info()
    sp = stream.cuda_stream
    out = {"workload": f"nmf_{m // 1000}k_{n // 1000}k_r{r}", "m": m, "n": n, "r": r,
           "data": "synthetic: X uniform on the grid k/256 (exact in bf16), V0, W0 uniform [0,1) FP32",
           "precision": "X bf16; V, W FP32 as 3 bf16 limbs on tcgen05 (kind::f16), FP32 accumulation; "
                        "Gram matrices FP64 from sums in pairs of floats",
           "limb_cols": info["limb_cols"], "stages": info["stages"]}
    iters = args.nmf_iters
    for algo in ("mult", "apg"):
        h.set_factors(V0, W0, sp)
        h.iterate(3, algo, 1e-10, sp)
        h.sync(sp)
        l0 = h.info()["launches"]
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        h.iterate(iters, algo, 1e-10, sp)
        e1.record(stream)
        torch.cuda.synchronize()
        h.sync(sp)
        ms = e0.elapsed_time(e1) / iters
        f = h.objective(sp)
        paper = NMF_PAPER_1GPU_S.get(r, {}).get(algo)
        out[algo] = {"iters_per_s": 1e3 / ms, "ms_per_iter": ms, "iters": iters,
                     "seconds_per_10000_iters": 10.0 * ms,
                     "paper_1gpu_seconds_per_10000_iters": paper,
                     "gpu_launches": int(h.info()["launches"] - l0), "objective_after": f}
    # roofline of the products: X (bf16) streamed once per launch, the limb panel and partial slots
    a_ms, b_ms = h.time_products(10, sp)
    xbytes = 2.0 * m * n
    pa = xbytes + info["limb_cols"] * n * 2 + 4.0 * r * m
    pb = xbytes + info["limb_cols"] * m * 2 + 4.0 * r * n
    peak, peak_kind = measured_peak_hbm()
    avg_ms = (a_ms + b_ms) / 2
    achieved = (pa + pb) / 2 / (avg_ms / 1e3) / 1e9
    flops = 2.0 * 128 * info["limb_cols"] * 64 * (info["units_xwt"] + info["units_vtx"]) / 2
    out["roofline"] = {"bound": "hbm", "kernel": "k_nmf_gemm (both products)", "achieved": achieved,
                       "peak": peak, "unit": "GB/s", "frac": achieved / peak, "peak_source": f"{peak_kind} hbm_gbs",
                       "ms_x_wt": a_ms, "ms_vt_x": b_ms, "bytes_per_launch": (pa + pb) / 2,
                       "tensor_tflops": flops / (avg_ms / 1e3) / 1e12, "traffic": nmf_traffic(m, n, r)}
    out["product_share_of_iteration"] = (a_ms + b_ms) / out["mult"]["ms_per_iter"]
    # end to end: host factors in, iterations, host factors out
    e2e_it = max(1, iters // 2)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    h.set_factors(V0, W0, sp)
    h.iterate(e2e_it, "mult", 1e-10, sp)
    Vh, Wh = h.factors(sp)
    e2e_s = time.perf_counter() - t0
    out["e2e"] = {"value": e2e_it / e2e_s, "unit": "iter/s", "iters": e2e_it,
                  "h2d_bytes": int(4 * r * (m + n)), "d2h_bytes": int(4 * r * (m + n)),
                  "timing": "wall clock: nmf_set_factors, nmf_iterate, nmf_get_factors (host arrays)"}
    h.close()
    if cpu_baseline:
        # the FP64 oracle as it stands (one thread), one multiplicative iteration
        # of the same workload
        import oracle
        oracle.build()
        t0 = time.perf_counter()
        oracle.nmf(X, V0, W0, 1, "mult", 1e-10)
        cs = time.perf_counter() - t0
        out["cpu_baseline"] = {"value": 1.0 / cs, "unit": "iter/s", "cores": 1, "kind": "oracle",
                               "sample": f"one multiplicative iteration of the full {m} x {n}, r = {r} workload "
                                         "(orc_nmf, FP64, one thread)"}
    return out


def run_ours(args, rank, world):
    import torch

    import synth
    from paper_2010_16114_gb300 import build
    from paper_2010_16114_gb300.cox import CoxProblem

    build()
    synth.build_device()
    local = int(os.environ.get("LOCAL_RANK", "0"))
    torch.cuda.set_device(local)
    if args.nmf_only:
        if rank == 0:
            print(json.dumps({"nmf": run_nmf(args, torch.cuda.current_stream(),
                                             cpu_baseline=world == 1 and not args.no_cpu_baseline)}), flush=True)
        return 0
    r = recipe(args)
    n, p, k = r.n, r.p, r.k
    stream = torch.cuda.current_stream()

    t_setup0 = time.perf_counter()
    w = synth.Workload(r)
    thr = torch.from_numpy(w.thr.view(np.int32).copy()).cuda()
    packed = torch.empty((n, (p + 3) // 4), dtype=torch.uint8, device="cuda")
    w.packed_rows_device(packed.data_ptr(), stream.cuda_stream, thr.data_ptr())
    torch.cuda.synchronize()
    prob = CoxProblem(packed, w.y, w.delta, p=p, precision=args.precision, tile_m=args.tile_m, stages=args.stages,
                      chunks=args.chunks, issue=args.issue, window=args.window)
    del packed, thr
    torch.cuda.empty_cache()
    lmax = prob.lambda_max()
    L = prob.lipschitz(tol=1e-4, maxiter=100)
    step = 1.0 / L
    lams = lmax * r.lambda_fracs()
    forced = args.tile_m or args.chunks or args.stages or args.issue
    tune = None if (args.no_autotune or forced) else prob.autotune(k, reps=2)
    t_setup = time.perf_counter() - t_setup0

    beta = prob.zeros(k)
    for _ in range(args.warmup):
        prob.prox_step(beta, lams, step)
    prob.sync()
    launches0 = prob.info()["launches"]
    clocks = Clocks(local)
    torch.cuda.synchronize()
    barrier(world)
    clocks.start()
    prob.profile(True)
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    torch.cuda.nvtx.range_push("timed")
    ev0.record(stream)
    for _ in range(args.steps):
        prob.prox_step(beta, lams, step)
    ev1.record(stream)
    torch.cuda.synchronize()
    torch.cuda.nvtx.range_pop()
    barrier(world)
    ms = ev0.elapsed_time(ev1)
    ck = clocks.stop()
    prob.profile(False)
    prob.sync()
    cls_ms, cls_n = prob.profile_read()
    pinfo = prob.info()
    launches = pinfo["launches"] - launches0
    F_last = prob.last_objective(k)
    ms_max = max_over_ranks(ms, world)
    ms_step = ms_max / args.steps
    value = world * args.steps / (ms_max / 1e3)

    # algorithmic bytes (packed X padded to 128 per dimension, as streamed by each product)
    xb = (-(-n // 128) * 128) * (-(-p // 128) * 128) / 4.0
    # limb bytes per coefficient: 8 e2m1 nibbles or 4 e4m3 bytes; 10 nibbles in the wide form
    plan = prob.plan(k)
    lb1, lb4 = (5 if plan[q]["form"] == "wide" else 4 for q in ("x_b", "xt_v"))
    b1 = xb + p * lb1 * k + k * n * 4              # X, beta limbs, eta partials
    b4 = xb + n * lb4 * k + 8 * k * p              # X, V limbs, beta read+write
    # scans, per subject and column: eta partials read (4), eta as a pair of floats, w and V written
    # and read once (16 + 8 + 8), event-group index and flags (7), limbs written
    scan_bytes = k * n * (43 + lb4)
    iter_bytes = b1 + b4 + scan_bytes + 12 * k * p  # + beta limbs / l1 pass
    gemm_ms = cls_ms[0] + cls_ms[1]
    gemm_n = cls_n[0] + cls_n[1]
    avg_launch_s = (gemm_ms / max(gemm_n, 1)) / 1e3
    achieved = ((b1 + b4) / 2.0) / avg_launch_s / 1e9
    peak, peak_kind = measured_peak_hbm()
    traffic = gemm_traffic(k, n, p, args.precision)

    # end to end: host buffers through the C ABI, copies inside the timed region
    e2e = None
    if args.e2e_steps > 0:
        beta_h = torch.zeros((k, p), dtype=torch.float32).pin_memory().numpy()
        beta_h[:] = beta.cpu().numpy()
        prob.prox_step_host(beta_h, lams, step)  # warm
        t0 = time.perf_counter()
        for _ in range(args.e2e_steps):
            prob.prox_step_host(beta_h, lams, step)
        e2e_s = time.perf_counter() - t0
        e2e_s = max_over_ranks(e2e_s, world)
        e2e = {"value": world * args.e2e_steps / e2e_s, "unit": UNIT, "h2d_bytes_per_step": int(k * p * 4 + k * 8),
               "d2h_bytes_per_step": int(k * p * 4 + 4), "steps": args.e2e_steps}

    # plain FP32 GEMV path on the same resident data
    gemv = None
    if not args.no_gemv and args.gemv_steps > 0:
        b0 = beta.clone()
        b_split = b0.clone()
        prob.prox_step(b_split, lams, step)
        prob.set_precision("fp32_gemv")
        b_gemv = b0.clone()
        prob.prox_step(b_gemv, lams, step)
        prob.sync()
        diff = float(torch.linalg.vector_norm(b_gemv - b_split) / max(torch.linalg.vector_norm(b_split), 1e-30))
        g0 = torch.cuda.Event(enable_timing=True)
        g1 = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        g0.record(stream)
        for _ in range(args.gemv_steps):
            prob.prox_step(b_gemv, lams, step)
        g1.record(stream)
        torch.cuda.synchronize()
        gms = g0.elapsed_time(g1) / args.gemv_steps
        g_hbm = 2 * k * xb / (gms / 1e3) / 1e9
        gemv = {"iters_per_s": 1e3 / gms, "ms_per_step": gms, "steps": args.gemv_steps,
                "lambda_iters_per_s": k * 1e3 / gms, "speedup_of_batched": (1e3 / ms_step) / (1e3 / gms),
                "hbm_gbs": g_hbm, "hbm_frac": g_hbm / peak,
                "rel_l2_vs_batched_one_step": diff}
        prob.set_precision(args.precision)

    # the path fit (Section 6 rule): every penalty from beta = 0 to
    # |F_t - F_{t-10}| / |F_t + 1| < tol or the iteration cap, 10 iterations at a time
    path = None
    if args.path_iters > 0:
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        Bpath, iters, obj, conv = prob.path_fit(lams, step, max_iter=args.path_iters, tol=args.path_tol)
        torch.cuda.synchronize()
        pt = time.perf_counter() - t0
        steps_run = int(np.max(iters))
        path = {"iters_per_s": steps_run / pt, "lambda_iters_per_s": k * steps_run / pt, "seconds": pt,
                "max_iter": args.path_iters, "tol": args.path_tol, "iterations_run": steps_run,
                "iterations_per_column": [int(x) for x in iters],
                "converged_columns": int(np.sum(np.asarray(iters) < args.path_iters)),
                "final_objective": [float(x) for x in obj],
                "timing": "wall clock around cox_path_fit (10 iterations at a time, host reads the "
                          "k objectives after each run of them), beta = 0 to the stopping rule or the cap"}

    # the active-set X B late in the path: the 8 largest penalties from the
    # path fit's coefficients, dense then with the active set, same iterations
    active = None
    if path is not None and args.active_steps > 0:
        ka = min(8, k)
        lam_a = lams[:ka]

        def timed(on):
            b = Bpath[:ka].clone()
            prob.set_active_set(on)
            prob.prox_step(b, lam_a, step)  # warm: plans, the active copy
            prob.sync()
            r0 = prob.info()["active_rebuilds"]
            prob.profile(True)
            a0 = torch.cuda.Event(enable_timing=True)
            a1 = torch.cuda.Event(enable_timing=True)
            a0.record(stream)
            for _ in range(args.active_steps):
                prob.prox_step(b, lam_a, step)
            a1.record(stream)
            torch.cuda.synchronize()
            prob.profile(False)
            prob.sync()
            cms, _ = prob.profile_read()
            inf = prob.info()
            split = {"x_b": cms[0] / args.active_steps, "xt_v_step": cms[1] / args.active_steps,
                     "scans": cms[2] / args.active_steps, "other_incl_active_set_work": cms[3] / args.active_steps}
            return a0.elapsed_time(a1) / args.active_steps, inf, split, inf["active_rebuilds"] - r0

        d_ms, _, d_split, _ = timed(False)
        a_ms, ainfo, a_split, a_reb = timed(True)
        prob.set_active_set(False)
        cols = ainfo["active_cols"]
        act_bytes = (-(-n // 128) * 128) * (-(-max(cols, 1) // 256) * 256) / 4.0 if cols >= 0 else xb
        active = {"lambdas": f"the {ka} largest of the grid, from the path fit's coefficients", "k": ka,
                  "active_cols": cols, "support_cols_limit": (-(-p // 1024) * 1024) // 4,
                  "dense_ms_per_step": d_ms, "active_ms_per_step": a_ms,
                  "dense_iters_per_s": 1e3 / d_ms, "active_iters_per_s": 1e3 / a_ms,
                  "x_b_bytes_per_iteration": {"dense": xb, "active": act_bytes},
                  "rebuilds": ainfo["active_rebuilds"], "rebuilds_in_timed_steps": a_reb,
                  "kernel_ms_per_step": {"dense": d_split, "active": a_split}, "steps": args.active_steps}

    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        cpu = OracleSample(r, args.cpu_sample_cols).baseline(args.cpu_sample_steps)

    prob.close()
    del beta
    torch.cuda.empty_cache()
    nmf = (run_nmf(args, stream, cpu_baseline=world == 1 and not args.no_cpu_baseline)
           if (rank == 0 and args.nmf_iters > 0) else None)
    if rank != 0:
        return 0
    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_step, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "e2m1" if args.precision == "split_e2m1" else "e4m3", "data": "synthetic",
        "precision": ("genotype products: codes and 8-limb split coefficients as e2m1 on tcgen05 "
                      "(kind::mxf4, unit block scales), FP32 accumulation; risk-set scans in pairs of floats per subject, FP64 per event time and in the objective"
                      if args.precision == "split_e2m1" else
                      "genotype products: codes and 4-limb split coefficients as e4m3 on tcgen05 "
                      "(kind::f8f6f4), FP32 accumulation; risk-set scans in pairs of floats per subject, FP64 per event time and in the objective"),
        "config": {"workload": workload_name(r), "n": n, "p": p, "k": k,
                   "l2": "inputs larger than L2: 2 x ~50 GB of packed genotypes streamed per step",
                   "parallelism": "replicas" if world > 1 else "single GPU",
                   "step_size": step, "lambda_max": lmax,
                   "pipeline": {"autotune": tune,
                                "x_b_in_use": {f: pinfo[f] for f in ("tile_m", "chunks", "stages", "ring", "issue")},
                                "xt_v_issue": pinfo["issue_xtv"]}},
        "lambda_iters_per_s": value * k,
        "hbm_gbs": iter_bytes / (ms_step / 1e3) / 1e9,
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s",
                     "frac": achieved / peak, "traffic": traffic,
                     "kernel": "k_packed_gemm (tensor-core genotype product, both launches per step)",
                     "peak_source": f"{peak_kind} hbm_gbs", "bytes_per_launch": (b1 + b4) / 2.0,
                     "avg_launch_ms": avg_launch_s * 1e3},
        "kernel_ms_per_step": {"x_b_product": cls_ms[0] / args.steps, "xt_v_product_step": cls_ms[1] / args.steps,
                               "scans": cls_ms[2] / args.steps, "other": cls_ms[3] / args.steps},
        "cpu_baseline": cpu,
        "path_fit": path,
        "active_set": active,
        "e2e": e2e,
        "gpu_launches": int(launches),
        "clocks": ck,
        "fp32_gemv": gemv,
        "nmf": nmf,
        "objective_last": [float(x) for x in F_last[:4]],
        "setup_s": t_setup,
    }
    print(json.dumps(line), flush=True)
    return 0


def main():
    args = parse()
    rank, world = dist_init(args)
    if args.impl == "reference":
        rc = run_reference(args, rank, world)
    else:
        rc = run_ours(args, rank, world)
    if world > 1:
        import torch.distributed as dist
        dist.destroy_process_group()
    return rc


if __name__ == "__main__":
    sys.exit(main())
