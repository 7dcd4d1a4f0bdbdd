"""Benchmark: quaternion pseudoinverse solves per second on one GB300.

Workload (one "step"): a full qpinv_solve of a square 2048 x 2048 quaternion
matrix A = U diag(sigma) V^H (U, V Haar quaternion unitaries, sigma
log-spaced from 1 to 1e-6) with QHPI19 in mixed precision: BF16-split
tensor-core products with FP32 accumulation, then FP64-residual polish
iterations, then the four Penrose residuals in FP64.  Inputs are resident in
HBM; A alone (134 MB of FP64 planes) exceeds the 129 MB L2, and every step
streams several times that through HBM.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Prints ONE JSON line (rank 0).  With --impl reference the FP64 CPU oracle is
timed on the host cores on a bounded sample of the same workload (rank 0
only; other ranks exit 0).
"""
import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "pinv solves/s & quaternion-GEMM TFLOP/s (% TC peak) to rel. Penrose res <=1e-10"
# Quaternion GEMMs of the workload's QHPI19 solve that the CPU-baseline
# sample extrapolates to: iterations x 7 products + 4 Penrose products.  The
# iteration count is the one the GPU arm reports for this workload
# ("iters" in its JSON line).
WORKLOAD_ITERS = 14


def peaks():
    path = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(path):
        with open(path) as f:
            p = json.load(f)
        return p.get("bf16_tflops", 1900.0), p.get("bf16_tflops_sustained", 1700.0), p.get("hbm_gbs", 6800.0), "measured"
    return 1900.0, 1700.0, 6800.0, "fallback"


class ClockSampler:
    """Samples nvidia-smi clocks and throttle reasons while running."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None
        self.lines = []

    def __enter__(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.Q,
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None
        return self

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def __exit__(self, *exc):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
            self.t.join(timeout=2)

    def summary(self):
        sm, mx, reasons = [], None, set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            f = [x.strip() for x in ln.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx = float(f[2])
            except ValueError:
                continue
            for nm, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": mx,
                "reasons": sorted(reasons), "samples": len(sm)}


def make_workload(n, device):
    """(A, U, sigma, V) of the square log-spaced workload."""
    from paper_2605_01464_gb300 import inputs
    return inputs.logspaced_square(n, 1e-6, seed_u=1, seed_v=2, device=device)


def oracle_pinv_error(X, U, sigma, V):
    """Relative Frobenius error of the GPU's X against the FP64 oracle's exact
    pseudoinverse V Sigma^-1 U^H of the generator's factors (CPU-baseline leg:
    runs on the host cores after the timed region)."""
    import numpy as np

    import oracle

    t0 = time.perf_counter()
    want = oracle.pinv_from_svd(U, sigma, V)
    X = np.asarray(X)
    err = float(np.linalg.norm(X - want) / np.linalg.norm(want))
    return err, time.perf_counter() - t0


def cpu_baseline_sample(A, iters, budget_s=30.0):
    """Times one QHPI19 iteration (7 quaternion GEMMs) of the FP64 oracle on
    the full-size input and extrapolates to a full solve of `iters`
    iterations plus the 4 Penrose products."""
    import numpy as np

    import oracle

    m, n = A.shape[1], A.shape[2]
    X0 = oracle.init_x0(A, oracle.alpha(A, "safe"))
    t0 = time.perf_counter()
    oracle.step(A, X0, "qhpi19")
    t_iter = time.perf_counter() - t0
    gemm_count = 7 * iters + 4
    t_solve = t_iter * gemm_count / 7.0
    return {"value": 1.0 / t_solve, "unit": "solves/s", "cores": os.cpu_count(), "kind": "oracle",
            "sample": "one QHPI19 iteration (7 quaternion GEMMs, %dx%d, FP64 oracle, %.1f s) extrapolated by "
                      "quaternion-GEMM count to %d iterations + 4 Penrose products" % (m, n, t_iter, iters),
            "sample_seconds": t_iter}


def run_reference(args, rank):
    if rank != 0:
        return 0
    import numpy as np  # noqa: F401

    from oracle import build as obuild
    obuild.build()
    A = make_workload(args.n, "cpu")[0]
    steps = []
    for k in range(args.warmup + args.steps):
        s = cpu_baseline_sample(A, WORKLOAD_ITERS)
        if k >= args.warmup:
            steps.append(s["sample_seconds"])
    t_iter = statistics.mean(steps)
    t_solve = t_iter * (7 * WORKLOAD_ITERS + 4) / 7.0
    value = 1.0 / t_solve
    line = {"metric": METRIC, "value": value, "unit": "solves/s", "n_gpus": args.gpus, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": t_iter * 1e3, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f64", "data": "synthetic", "impl": "reference",
            "config": workload_config(args),
            "cpu_baseline": {"value": value, "unit": "solves/s", "cores": os.cpu_count(), "kind": "oracle",
                             "sample": "each step: one QHPI19 iteration (7 quaternion GEMMs) of the FP64 oracle "
                                       "on the full %dx%d input, extrapolated to %d iterations + 4 Penrose "
                                       "products" % (args.n, args.n, WORKLOAD_ITERS)},
            "e2e": {"value": value, "unit": "solves/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


def kernel_qgemm(args, torch, qpinv):
    """Times the tcgen05 quaternion GEMM alone on seeded n x n operands."""
    from paper_2605_01464_gb300 import inputs
    n = args.n
    A = torch.from_numpy(inputs.gaussian_quaternion(n, n, 21)).cuda()
    B = torch.from_numpy(inputs.gaussian_quaternion(n, n, 22)).cuda()
    ctx = qpinv.Context(0, profile=True)
    ctx.configure(emu_pair={"auto": "auto", "0": False, "1": True}[args.emu_pair])
    prec = args.gemm_precision
    for _ in range(args.warmup):
        ctx.qgemm(A, B, precision=prec, split_level=args.split)
    ctx.reset_stats()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        ctx.qgemm(A, B, precision=prec, split_level=args.split)
    torch.cuda.synchronize()
    wall = (time.perf_counter() - t0) / args.steps
    st = ctx.stats()
    key = "emu" if st["emu_gemm_launches"] else "tc"
    launches = max(st["%s_gemm_launches" % key], 1)
    gms = st["%s_gemm_ms" % key]
    kname = "k_qgemm_tc"
    if key == "emu":
        kname = "k_qgemm_emu"
    print(json.dumps({"kernel": kname, "n": n, "precision": prec,
                      "split": args.split, "launches_per_product": launches / args.steps, "ms_per_launch": gms / launches,
                      "gemm_ms_per_product": gms / args.steps,
                      "all_kernels_ms_per_product": (gms + st["ew_ms"]) / args.steps,
                      "wall_ms_per_product": wall * 1e3,
                      "tflops_algorithmic": st["%s_gemm_flops" % key] / gms / 1e9,
                      "tflops_issued": st["%s_gemm_flops_issued" % key] / gms / 1e9}))
    return 0


def gemm_target_records(torch, qpinv, local, sizes=(4096, 8192), warmup=2, reps=5):
    """Roofline entries of the single-pass BF16 tensor-core quaternion GEMM
    (k_qgemm_tc, one BF16 term per operand) at n x n x n, n >= 4096: the
    kernel's own CUDA-event time per launch (library events on the launch
    stream), 32 flops per quaternion multiply-add, against the measured BF16
    burst peak (a kernel timed alone), with the clocks sampled meanwhile."""
    bf16_burst, _, _, src = peaks()
    out = []
    gen = torch.Generator(device="cuda:%d" % local)
    for n in sizes:
        gen.manual_seed(7000 + n)
        A = torch.randn((4, n, n), dtype=torch.float64, device="cuda:%d" % local, generator=gen)
        B = torch.randn((4, n, n), dtype=torch.float64, device="cuda:%d" % local, generator=gen)
        C = torch.empty_like(A)
        ctx = qpinv.Context(local, profile=True)
        for _ in range(warmup):
            ctx.qgemm(A, B, precision="tc", split_level=1, C=C)
        torch.cuda.synchronize()
        ctx.reset_stats()
        with ClockSampler(local) as clk:
            for _ in range(reps):
                ctx.qgemm(A, B, precision="tc", split_level=1, C=C)
            torch.cuda.synchronize()
        st = ctx.stats()
        ctx.close()
        launches = max(st["tc_gemm_launches"], 1)
        ms = st["tc_gemm_ms"] / launches
        alg = 32.0 * n ** 3 / (ms * 1e-3) / 1e12
        out.append({"bound": "tensor", "achieved": alg, "peak": bf16_burst, "unit": "TFLOP/s",
                    "frac": alg / bf16_burst, "traffic": None,
                    "kernel": "k_qgemm_tc (single-pass BF16 quaternion GEMM, %d x %d x %d)" % (n, n, n),
                    "launches": launches, "ms_per_launch": ms, "achieved_issued": alg, "frac_issued": alg / bf16_burst,
                    "peak_source": "%s bf16_tflops burst (MEASURED_PEAKS.json): the kernel is timed alone" % src,
                    "clocks": clk.summary()})
        del A, B, C
        torch.cuda.empty_cache()
    return out


# CTA GEMM engines of qpinv_solve_batched by index (qpinv_options.batched_tile)
BATCH_ENGINES = ["16x16", "32x32", "64x32", "32x64", "64x64", "tc (tensor-core exact slices)"]


def batched_flops(m, n, method, steps):
    """Algorithmic flops of one batched solve: 32 per quaternion multiply-add
    of every product -- per iteration the method's products on the residual
    side s = min(m, n) (QHPI19: 2 s^2 l + 5 s^3 with l = max(m, n); QSAI
    2 s^2 l + 4 s^3; NS 2 s^2 l) -- plus the 4 Penrose products 2 m n (m + n)."""
    s, l = min(m, n), max(m, n)
    per = {"qhpi19": 2 * s * s * l + 5 * s ** 3, "qsai": 2 * s * s * l + 4 * s ** 3, "ns": 2 * s * s * l}
    return 32.0 * (steps * per.get(method, per["qhpi19"]) + 2.0 * m * n * (m + n))


def bench_batched(args, torch, qpinv, world=1, rank=0, local=0):
    """4096 pure-quaternion blocks (m, n ~ U[16, 256], rank ~ U[4, min(m, n)])
    solved by qpinv_solve_batched in one persistent launch per step.  With N
    ranks each GPU solves its own 4096 blocks (weak scaling; no collective on
    the data path, only the timing reduction)."""
    import numpy as np

    from paper_2605_01464_gb300 import inputs
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    count = args.batch_count
    mats = inputs.pure_quaternion_batch(count, seed=3 + 1000 * rank)
    As = [torch.from_numpy(a).cuda() for a in mats]
    Xs = [torch.empty((4, a.shape[2], a.shape[1]), dtype=torch.float64, device="cuda") for a in As]
    ctx = qpinv.Context(local)
    for _ in range(args.warmup):
        ctx.solve_batched(As, args.method, tol=args.tol, max_iter=200, Xs=Xs)
    torch.cuda.synchronize()
    tune_ms = ctx.stats()["batched_tune_ms"]
    ctx.reset_stats()
    if dist:
        dist.barrier()
    t0 = time.perf_counter()
    with ClockSampler(local) as clk:
        for _ in range(args.steps):
            _, infos = ctx.solve_batched(As, args.method, tol=args.tol, max_iter=200, Xs=Xs)
        torch.cuda.synchronize()
    dt, solves = reduce_timing(time.perf_counter() - t0, count * args.steps, dist, "cuda")
    if dist:
        dist.destroy_process_group()
    if rank != 0:
        return 0
    e1 = [i["E_rel"][0] for i in infos]
    its = [i["iters"] for i in infos]
    st = ctx.stats()
    # steps computed per matrix: the returned iterations plus the rejected
    # step of a plateau stop
    flops = sum(batched_flops(a.shape[1], a.shape[2], args.method, i["iters"] + (i["status"] == "plateau"))
                for a, i in zip(mats, infos))
    bf16_burst, bf16_sust, _, src = peaks()
    ach = flops / (dt / args.steps) / 1e12
    roof = {"bound": "tensor", "achieved": ach, "peak": bf16_sust, "unit": "TFLOP/s", "frac": ach / bf16_sust,
            "traffic": None, "kernel": "the persistent batched kernel (%s engine), whole call" %
                                       BATCH_ENGINES[st["batched_tile"]],
            "algorithmic_flops_per_step": flops,
            "peak_source": "%s bf16_tflops_sustained (MEASURED_PEAKS.json)" % src}
    cpu = None
    if world == 1 and not args.no_cpu_baseline:
        import oracle
        sample = list(range(0, count, max(1, count // 16)))[:16]  # 16 evenly spaced blocks
        t0 = time.perf_counter()
        errs = []
        for b in sample:
            xo, _ = oracle.solve(mats[b], args.method, tol=args.tol, max_iter=200)
            errs.append(float(np.linalg.norm(Xs[b].cpu().numpy() - xo) / np.linalg.norm(xo)))
        t_cpu = time.perf_counter() - t0
        cpu = {"value": len(sample) / t_cpu, "unit": "solves/s", "cores": os.cpu_count(), "kind": "oracle",
               "sample": "the FP64 oracle's %s on 16 evenly spaced blocks of the batch (%.1f s); the GPU X of "
                         "those blocks against the oracle's: max relative error %.2e"
                         % (args.method, t_cpu, max(errs)),
               "x_relerr_vs_oracle_max": max(errs)}
    print(json.dumps({"metric": "batched pinv solves/s", "value": solves / dt, "unit": "solves/s",
                      "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "ms_per_step": dt / args.steps * 1e3,
                      "higher_is_better": True, "scaling": "weak",
                      "dtype": "df32 masters (double-FP32); tc engine: exact 7-bit BF16 slices",
                      "data": "synthetic",
                      "config": {"workload": "%d pure-quaternion blocks, m, n ~ U[16,256], rank ~ U[4,min(m,n)], "
                                             "seed 3, %s, rel. tol %g, one persistent kernel per step replayed as a "
                                             "captured CUDA graph, autotuned CTA GEMM tile"
                                             % (count, args.method, args.tol),
                                 "tile": BATCH_ENGINES[st["batched_tile"]],
                                 "autotune_ms": tune_ms, "graph_replays": st["batched_graph_replays"]},
                      "gpu_launches": st["kernel_launches"], "roofline": roof, "cpu_baseline": cpu,
                      "result": {"max_E1_rel": max(e1), "median_iters": sorted(its)[len(its) // 2],
                                 "statuses": sorted(set(i["status"] for i in infos))},
                      "clocks": clk.summary()}), flush=True)
    return 0


def _timed_solve(ctx, torch, A, method, tol, max_iter=500):
    """One solve on the current stream, timed with CUDA events."""
    stream = torch.cuda.current_stream()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    e0.record(stream)
    _, info = ctx.solve(A, method, tol=tol, max_iter=max_iter, stream=stream)
    e1.record(stream)
    torch.cuda.synchronize()
    return e0.elapsed_time(e1), info


def bench_rankdef(args, torch, qpinv):
    """Rank-2048 8192 x 4096 A = QL diag(sigma) QR^H, sigma geometric 1..1e-4
    (seeds 4, 5): QHPI19 and Newton-Schulz to the plateau stop, each with
    FP64-accurate tensor-core products throughout (EMU) and in the default
    mixed precision (BF16-split bulk with FP64-accurate polish; a result that
    fails the Penrose check is repeated in EMU, and the line says which
    precision produced X).  One step = one QHPI19 EMU solve.  Every X is
    compared with the FP64 oracle's exact pseudoinverse QR Sigma^-1 QL^H of
    the generator's factors (CPU-baseline leg, after the timed solves)."""
    import numpy as np

    from paper_2605_01464_gb300 import inputs
    dev = "cuda" if args.gen_device == "cuda" else "cpu"
    A_host, QL, sig, QR = inputs.rank_deficient(8192, 4096, 2048, 1e-4, 4, 5, device=dev)
    A = torch.from_numpy(A_host).cuda()
    ctx = qpinv.Context(0, precision="emu", profile=True)
    out, Xs = {}, {}
    with ClockSampler(0) as clk:
        for method in ("qhpi19", "ns"):
            for prec in ("emu", "mixed"):
                ctx.configure(precision=prec)
                for _ in range(args.warmup if (method, prec) == ("qhpi19", "emu") else 0):
                    _timed_solve(ctx, torch, A, method, args.tol)
                ctx.reset_stats()
                times, info = [], None
                for _ in range(args.steps if (method, prec) == ("qhpi19", "emu") else 1):
                    stream = torch.cuda.current_stream()
                    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    torch.cuda.synchronize()
                    e0.record(stream)
                    X, info = ctx.solve(A, method, tol=args.tol, max_iter=500, stream=stream)
                    e1.record(stream)
                    torch.cuda.synchronize()
                    times.append(e0.elapsed_time(e1))
                st = ctx.stats()
                key = "%s_%s" % (method, prec)
                Xs[key] = X.cpu().numpy()
                out[key] = {"ms_per_solve": statistics.mean(times), "iters": info["iters"],
                            "status": info["status"], "precision_of_X": info["precision"],
                            "E_rel": info["E_rel"], "gemms": info["gemms"], "gpu_launches": st["kernel_launches"],
                            "roofline": kernel_rooflines(st)}
    cpu = None
    if not args.no_cpu_baseline:
        import oracle
        t0 = time.perf_counter()
        want = oracle.pinv_from_svd(QL, sig, QR)
        t_ref = time.perf_counter() - t0
        for key, X in Xs.items():
            out[key]["x_relerr_vs_oracle"] = float(np.linalg.norm(X - want) / np.linalg.norm(want))
        cpu = {"value": 1.0 / t_ref, "unit": "reference pseudoinverses/s", "cores": os.cpu_count(), "kind": "oracle",
               "sample": "the FP64 oracle's QR Sigma^-1 QL^H of the generator's factors (one 4096 x 2048 x 8192 "
                         "quaternion product, %.1f s), the reference of x_relerr_vs_oracle" % t_ref}
    q = out["qhpi19_emu"]
    print(json.dumps({
        "metric": "rank-deficient pinv solves/s to rel. Penrose res (FP64 floor)", "value": 1e3 / q["ms_per_solve"],
        "unit": "solves/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "ms_per_step": q["ms_per_solve"],
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "exact-slice bf16 (FP64-accurate)",
        "data": "synthetic",
        "config": {"workload": "8192x4096 quaternion, rank 2048, A = QL diag(sigma) QR^H, sigma geometric 1..1e-4, "
                               "orthonormal factors from Gaussian quaternion matrices (seeds 4, 5); left residual "
                               "(4096 side); EMU and mixed precision; rel. tol %g with plateau stop" % args.tol,
                   "l2": "inputs exceed L2"},
        "roofline": q["roofline"][0], "result": out, "cpu_baseline": cpu, "clocks": clk.summary()}), flush=True)
    return 0


# Example 3's table (n = 800, CPU seconds): QHPI19 6.188, QSAI 6.594,
# QHONSchultz(19) 13.87, QHONSchultz(10) 11.05.
PAPER_EX3_SECONDS = {"qhpi19": 6.188, "qsai": 6.594, "qhpim19": 13.87, "qhpim10": 11.05}


def bench_hyper(args, torch, qpinv):
    """Example 3: factorized (QHPI19, QSAI) against unfactorized hyperpower
    iterations (QHPIM of order 19 and 10, the example's QHONSchultz) on n x n
    Gaussian quaternion matrices (every component N(0, 1), seed 0), stop at
    ||X_{j+1} - X_j||_F <= 1e-10 as in the example; n = 800 with its fixed
    alpha = 7.8798e-5, n = 2048 with alpha = 1 / sigma_1^2 (power iteration,
    outside the timed region).  Mixed precision, and at n = 800 also every
    product FP64-accurate (EMU, the counterpart of the example's FP64
    arithmetic, where all products cost the same).  One step = one solve of
    each solver; the line's value is QHPIM(19) at n = 800, mixed precision."""
    from paper_2605_01464_gb300 import inputs
    solvers = (("qhpi19", "qhpi19", 19), ("qsai", "qsai", 10), ("qhpim19", "qhpim", 19), ("qhpim10", "qhpim", 10))
    out, roof = {}, None
    with ClockSampler(0) as clk:
        for n, precision, key in ((800, "mixed", "800"), (800, "emu", "800_emu"), (2048, "mixed", "2048")):
            A = torch.from_numpy(inputs.gaussian_quaternion(n, n, 0)).cuda()
            ctx = qpinv.Context(0, precision=precision, stop="paper_abs", profile=True)
            if n == 800:
                ctx.configure(alpha="user", alpha_user=7.8798e-5)
            else:
                ctx.configure(alpha="spectral")
                _, info = ctx.solve(A, "ns", tol=1.0, max_iter=1)
                ctx.configure(alpha="user", alpha_user=info["alpha"])
            res = {}
            for name, method, k in solvers:
                ctx.configure(hyper_order=k)
                for _ in range(args.warmup):
                    _timed_solve(ctx, torch, A, method, 1e-10, max_iter=100)
                ctx.reset_stats()
                times = []
                for _ in range(args.steps):
                    ms, info = _timed_solve(ctx, torch, A, method, 1e-10, max_iter=100)
                    times.append(ms)
                st = ctx.stats()
                res[name] = {"ms_per_solve": statistics.mean(times), "iters": info["iters"],
                             "status": info["status"], "E": info["E"], "gemms": info["gemms"],
                             "alpha": info["alpha"], "gpu_launches": st["kernel_launches"] // args.steps}
                if key == "800" and name == "qhpim19":
                    roof = kernel_rooflines(st)[0]
            res["time_ratio_order19"] = res["qhpim19"]["ms_per_solve"] / res["qhpi19"]["ms_per_solve"]
            res["time_ratio_order10"] = res["qhpim10"]["ms_per_solve"] / res["qsai"]["ms_per_solve"]
            out[key] = res
            ctx.close()
    paper = {"time_ratio_order19": PAPER_EX3_SECONDS["qhpim19"] / PAPER_EX3_SECONDS["qhpi19"],
             "time_ratio_order10": PAPER_EX3_SECONDS["qhpim10"] / PAPER_EX3_SECONDS["qsai"],
             "iters": {"qhpi19": 8, "qsai": 10, "qhpim19": 8, "qhpim10": 10}}
    q = out["800"]["qhpim19"]
    print(json.dumps({
        "metric": "unfactorized hyperpower QHONSchultz(19) solves/s (Example 3)", "value": 1e3 / q["ms_per_solve"],
        "unit": "solves/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "ms_per_step": q["ms_per_solve"],
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16-split/exact-slice (mixed)",
        "data": "synthetic",
        "config": {"workload": "n x n Gaussian quaternion matrices (components N(0,1), seed 0), n = 800 (alpha "
                               "7.8798e-5) and 2048 (alpha = 1/sigma_1^2); QHPI19, QSAI, QHPIM(19), QHPIM(10); "
                               "mixed precision (and EMU at n = 800); stop ||X_{j+1} - X_j||_F <= 1e-10",
                   "l2": "inputs of 20 MB (n = 800) fit in L2; no flush between solves"},
        "roofline": roof, "result": out, "paper_example3": paper, "clocks": clk.summary()}), flush=True)
    return 0


def _ssim(X, ref):
    """Mean structural similarity over the colour planes (Gaussian window,
    standard deviation 1.5, 11 x 11; constants (0.01)^2 and (0.03)^2 for a
    peak of 1), or None without scipy."""
    import numpy as np
    try:
        from scipy.ndimage import gaussian_filter
    except ImportError:
        return None
    vals = []
    for p in (1, 2, 3):
        x, y = X[p], ref[p]
        g = lambda a: gaussian_filter(a, 1.5, truncate=3.5)
        mx, my = g(x), g(y)
        sxx, syy, sxy = g(x * x) - mx * mx, g(y * y) - my * my, g(x * y) - mx * my
        c1, c2 = 0.01 ** 2, 0.03 ** 2
        vals.append(np.mean((2 * mx * my + c1) * (2 * sxy + c2) / ((mx * mx + my * my + c1) * (sxx + syy + c2))))
    return float(np.mean(vals))


def bench_cur(args, torch, qpinv):
    """CUR image completion (Sec. 5.1): a 512 x 768 synthetic colour image
    (seed 16) with 70 % of the pixels removed (seed 17), rank-60 CUR with
    U = C_J^+ C R_I^+, 25 iterations with fresh index sets (seed 18), Gaussian
    filter sigma = 0.5, QHPI19 pseudoinverses (rel. tol 1e-12) in mixed and
    in FP64 precision, the faster reported.  One step = one whole completion;
    the CPU baseline runs the FP64 oracle on the same completion."""
    import numpy as np
    from paper_2605_01464_gb300 import inputs
    m, n, r, T = 512, 768, 60, 25
    A = inputs.synthetic_rgb_image(m, n, 16)
    mask = inputs.completion_mask(m, n, 0.3, 17)
    Is, Js = inputs.cur_index_sets(m, n, r, T, 18)
    M = A * mask
    Md, maskd = torch.from_numpy(M).cuda(), torch.from_numpy(mask).cuda()
    stream = torch.cuda.current_stream()
    # The inner pseudoinverses are small (residual side 60): they are timed in
    # the default mixed precision and in FP64 (CUDA-core products, fewer
    # launches per product); the line reports the faster.  Timing runs have
    # kernel profiling off; one extra profiled completion gives the kernel
    # figures.
    timing = {}
    with ClockSampler(0) as clk:
        for prec in ("mixed", "fp64"):
            ctx = qpinv.Context(0, precision=prec)

            def run(Mx, mx):
                return ctx.cur_complete(Mx, mx, Is, Js, args.method, tol=1e-12, max_iter=200, sigma=0.5,
                                        stream=stream)

            for _ in range(args.warmup):
                run(Md, maskd)
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record(stream)
            for _ in range(args.steps):
                C, info = run(Md, maskd)
            e1.record(stream)
            torch.cuda.synchronize()
            ms = e0.elapsed_time(e1) / args.steps
            # end to end: host image, mask and result (pinned), copies in the timed region
            Mh = torch.from_numpy(M).pin_memory().numpy()
            mh = torch.from_numpy(mask).pin_memory().numpy()
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            for _ in range(args.steps):
                Ch, _ = run(Mh, mh)
            torch.cuda.synchronize()
            ms_e2e = (time.perf_counter() - t0) * 1e3 / args.steps
            ctx.configure(profile=True)
            ctx.reset_stats()
            run(Md, maskd)
            st = ctx.stats()
            ctx.close()
            timing[prec] = (ms, ms_e2e, st, C, info)
    best = min(timing, key=lambda k: timing[k][0])
    ms, ms_e2e, st, C, info = timing[best]
    C = C.cpu().numpy()
    mse = np.mean((C[1:] - A[1:]) ** 2)
    psnr = 10 * math.log10(1.0 / mse)
    base = None
    if not args.no_cpu_baseline:
        from oracle import cur as ocur
        t0 = time.perf_counter()
        Co, _ = ocur.cur_complete(M, mask, Is, Js, args.method, tol=1e-12, max_iter=200, sigma=0.5)
        t_cpu = time.perf_counter() - t0
        base = {"value": 1.0 / t_cpu, "unit": "completions/s", "cores": 1, "kind": "oracle",
                "sample": "the whole completion (25 iterations, 512x768, rank 60) by the FP64 oracle, %.1f s" % t_cpu,
                "max_rel_diff_vs_gpu": float(np.linalg.norm(C - Co) / np.linalg.norm(Co))}
    print(json.dumps({
        "metric": "CUR image completions/s (512x768, 70% missing, rank 60, 25 iterations)", "value": 1e3 / ms,
        "unit": "completions/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": "512x768 synthetic colour image (pure quaternions), 70%% of pixels removed, CUR rank 60 "
                               "with U = C_J^+ C R_I^+, 25 impute-reconstruct iterations, Gaussian filter 0.5, "
                               "%s pseudoinverses (%s precision, rel. tol 1e-12)" % (args.method.upper(), best),
                   "precision_ms": {k: v[0] for k, v in timing.items()},
                   "l2": "working set of 19 MB per image plane set fits in L2; no flush"},
        "e2e": {"value": 1e3 / ms_e2e, "unit": "completions/s", "h2d_bytes_per_step": M.nbytes + mask.nbytes,
                "d2h_bytes_per_step": C.nbytes},
        "gpu_launches": st["kernel_launches"],
        "roofline": kernel_rooflines(st)[0], "cpu_baseline": base,
        "result": {"psnr_db": psnr, "psnr_masked_db": 10 * math.log10(1.0 / np.mean((M[1:] - A[1:]) ** 2)),
                   "ssim": _ssim(C, A), "pinv": info, "paper_kodim16": {"psnr_db": 27.91, "ssim": 0.8126,
                                                                         "cpu_seconds": 150.39}},
        "clocks": clk.summary()}), flush=True)
    return 0


# Sec. 5.2's table (CPU seconds; QSVD, QNS, QSAI) per step size.
PAPER_LORENZ_SECONDS = {0.01: (994.45, 254.35, 74.34), 0.02: (115.61, 37.27, 10.21), 0.03: (35.34, 14.71, 4.22),
                        0.04: (15.11, 6.19, 1.70), 0.05: (6.89, 3.29, 0.98)}


def bench_filter(args, torch, qpinv):
    """Quaternion filtering of Lorenz signals (Sec. 5.2): for each step size
    dt in 0.01 .. 0.05 over [0, 40] (N = 40/dt + 1 samples, delay tau = 1,
    noise 0.5 per component), the (p+1) x (p+1) data matrix with p = (N-1)/2,
    h = X^+ s by QSAI and by Newton-Schulz (MIXED, rel. tol 1e-12), s_hat =
    X h and its error.  One step = one filter design at dt = 0.01 (2001 x 2001)
    with QSAI; the other cases are timed the same way and reported."""
    import numpy as np
    from paper_2605_01464_gb300 import inputs
    ctx = qpinv.Context(0, profile=True)
    stream = torch.cuda.current_stream()
    out, roof, line = {}, None, None
    with ClockSampler(0) as clk:
        for dt in (0.01, 0.02, 0.03, 0.04, 0.05):
            x, s = inputs.lorenz_signals(dt=dt)
            p = (x.shape[1] - 1) // 2
            xd, sd = torch.from_numpy(x).cuda(), torch.from_numpy(s).cuda()
            res = {"p": p}
            for method in ("qsai", "ns"):
                for _ in range(args.warmup):
                    ctx.toeplitz_filter(xd, sd, p, method=method, tol=1e-12, max_iter=2000, stream=stream)
                ctx.reset_stats()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize()
                e0.record(stream)
                for _ in range(args.steps):
                    h, sh, err, info = ctx.toeplitz_filter(xd, sd, p, method=method, tol=1e-12, max_iter=2000,
                                                           stream=stream)
                e1.record(stream)
                torch.cuda.synchronize()
                ms = e0.elapsed_time(e1) / args.steps
                st = ctx.stats()
                res[method] = {"ms": ms, "err": err, "iters": info["iters"], "status": info["status"],
                               "E1_rel": info["E_rel"][0], "gpu_launches": st["kernel_launches"] // args.steps}
                if dt == 0.01 and method == "qsai":
                    roof = kernel_rooflines(st)[0]
                    line = (ms, st["kernel_launches"] // args.steps)
                    xh = torch.from_numpy(x).pin_memory().numpy()
                    shh = torch.from_numpy(s).pin_memory().numpy()
                    torch.cuda.synchronize()
                    t0 = time.perf_counter()
                    for _ in range(args.steps):
                        ctx.toeplitz_filter(xh, shh, p, method=method, tol=1e-12, max_iter=2000, stream=stream)
                    torch.cuda.synchronize()
                    res["e2e_ms"] = (time.perf_counter() - t0) * 1e3 / args.steps
                    e2e_bytes = (x.nbytes + s.nbytes, 2 * 4 * 8 * (p + 1))
            res["paper_cpu_seconds_qsvd_qns_qsai"] = PAPER_LORENZ_SECONDS[dt]
            out[str(dt)] = res
    base = None
    if not args.no_cpu_baseline:
        from oracle import lorenz
        x, s = inputs.lorenz_signals(dt=0.05)
        p5 = (x.shape[1] - 1) // 2
        t0 = time.perf_counter()
        lorenz.design(x, s, p5, p5, "qsai", tol=1e-12, max_iter=2000)
        t5 = time.perf_counter() - t0
        scale = (2001.0 / (p5 + 1)) ** 3
        base = {"value": 1.0 / (t5 * scale), "unit": "designs/s", "cores": 1, "kind": "oracle",
                "sample": "QSAI design at dt = 0.05 (401 x 401) by the FP64 oracle, %.2f s, extrapolated by "
                          "(2001/401)^3 to dt = 0.01" % t5}
    ms, launches = line
    print(json.dumps({
        "metric": "Lorenz quaternion filter designs/s (dt 0.01: 2001x2001 data matrix, QSAI)", "value": 1e3 / ms,
        "unit": "designs/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "bf16-split/exact-slice (mixed)",
        "data": "synthetic",
        "config": {"workload": "Lorenz system (sigma 10, delta 8/3, gamma 28, start (1,1,1)) sampled at dt over "
                               "[0, 40] by RK4, delay tau = 1, purely imaginary noise N(0, 0.25) per component; "
                               "square Toeplitz data matrix of half the samples; h = X^+ s, QSAI, mixed precision",
                   "l2": "one 2001^2 quaternion matrix is 128 MB of FP64 planes, about L2: no flush"},
        "e2e": {"value": 1e3 / out["0.01"]["e2e_ms"], "unit": "designs/s", "h2d_bytes_per_step": e2e_bytes[0],
                "d2h_bytes_per_step": e2e_bytes[1]},
        "gpu_launches": launches, "roofline": roof, "cpu_baseline": base, "result": out,
        "clocks": clk.summary()}), flush=True)
    return 0


# Example 4's table: (IT, seconds) of Gl-QFOM, Gl-QGMRES, preconditioned Gl-QFOM, preconditioned Gl-QGMRES.
PAPER_KRYLOV = {3: ((697, 10.94), (697, 10.71), (308, 2.07), (244, 1.29)),
                6: ((1268, 50.56), (1264, 49.98), (542, 8.78), (419, 5.16)),
                9: ((1756, 278.15), (1752, 140.89), (746, 24.00), (568, 13.27)),
                12: ((2218, 449.83), (2212, 265.02), (951, 47.64), (703, 23.99))}


def bench_krylov(args, torch, qpinv):
    """Example 4 (Sec. 3.5): A X = B with A = A_s (1 - i + 2j + 1.5k), A_s the
    238 x 238 reservoir operator standing in for saylr1, B with uniform
    entries and m = 3, 6, 9, 12 columns; Gl-QFOM and Gl-QGMRES, plain and left
    preconditioned by QSAI (2 iterations), unrestarted, X_0 = 0, RR <= 1e-6,
    at most 3000 steps.  One step = one preconditioned Gl-QGMRES solve at
    m = 3 (the line's value); the rest are timed the same way and reported."""
    import numpy as np
    from paper_2605_01464_gb300 import inputs
    ctx = qpinv.Context(0)  # timing with kernel profiling off; one profiled solve for the kernel figures
    stream = torch.cuda.current_stream()
    variants = (("fom", "fom", 0), ("gmres", "gmres", 0), ("prec_fom", "fom", 2), ("prec_gmres", "gmres", 2))
    out, line = {}, None
    _, _, hbm, src = peaks()
    with ClockSampler(0) as clk:
        for m in (3, 6, 9, 12):
            A, B = inputs.krylov_system(m)
            Ad, Bd = torch.from_numpy(A).cuda(), torch.from_numpy(B).cuda()
            res = {}
            for name, kind, pk in variants:
                steps = args.steps if (m == 3 and name == "prec_gmres") else 1
                for _ in range(args.warmup if steps > 1 else 1):
                    ctx.global_krylov(Ad, Bd, kind, precond_iters=pk, tol=1e-6, max_iter=3000, stream=stream)
                ctx.reset_stats()
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize()
                e0.record(stream)
                for _ in range(steps):
                    X, info = ctx.global_krylov(Ad, Bd, kind, precond_iters=pk, tol=1e-6, max_iter=3000,
                                                stream=stream)
                e1.record(stream)
                torch.cuda.synchronize()
                ms = e0.elapsed_time(e1) / steps
                st = ctx.stats()
                res[name] = {"ms": ms, "iters": info["iters"], "converged": info["converged"],
                             "rel_res": info["rel_res"], "true_rel_res": info["true_rel_res"],
                             "gpu_launches": st["kernel_launches"] // steps}
                if m == 3 and name == "prec_gmres":
                    ctx.configure(profile=True)
                    ctx.reset_stats()
                    ctx.global_krylov(Ad, Bd, kind, precond_iters=pk, tol=1e-6, max_iter=3000, stream=stream)
                    st = ctx.stats()
                    ctx.configure(profile=False)
                    steps_prof = 1
                    gbs = st["ew_bytes"] / (st["ew_ms"] * 1e-3) / 1e9 if st["ew_ms"] > 0 else None
                    roof = {"bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s",
                            "frac": gbs / hbm if gbs else None, "traffic": None,
                            "kernel": "global Gram-Schmidt / update kernels (k_arnoldi, or k_block_dot, "
                                      "k_block_combine, k_norm_scale; bytes counted per launch)",
                            "ew_ms_per_solve": st["ew_ms"] / steps_prof,
                            "f64_gemm_ms_per_solve": st["f64_gemm_ms"] / steps_prof,
                            "peak_source": "%s hbm_gbs (MEASURED_PEAKS.json)" % src}
                    line = (ms, st["kernel_launches"] // steps_prof, roof)
                    Ah = torch.from_numpy(A).pin_memory().numpy()
                    Bh = torch.from_numpy(B).pin_memory().numpy()
                    torch.cuda.synchronize()
                    t0 = time.perf_counter()
                    for _ in range(steps):
                        ctx.global_krylov(Ah, Bh, kind, precond_iters=pk, tol=1e-6, max_iter=3000, stream=stream)
                    torch.cuda.synchronize()
                    e2e = ((time.perf_counter() - t0) * 1e3 / steps, A.nbytes + B.nbytes, B.nbytes)
            res["paper_it_seconds"] = dict(zip([v[0] for v in variants], PAPER_KRYLOV[m]))
            out[str(m)] = res
    base = None
    if not args.no_cpu_baseline:
        from oracle import krylov
        A, B = inputs.krylov_system(3)
        t0 = time.perf_counter()
        krylov.global_krylov(A, B, "gmres", precond_iters=2, tol=1e-6, max_iter=3000)
        t_cpu = time.perf_counter() - t0
        base = {"value": 1.0 / t_cpu, "unit": "solves/s", "cores": 1, "kind": "oracle",
                "sample": "one preconditioned Gl-QGMRES solve at m = 3 by the FP64 oracle, %.1f s" % t_cpu}
    ms, launches, roof = line
    print(json.dumps({
        "metric": "QSAI-preconditioned Gl-QGMRES solves/s (238x238 reservoir operator, m = 3, RR 1e-6)",
        "value": 1e3 / ms, "unit": "solves/s", "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
        "data": "synthetic",
        "config": {"workload": "A = A_s (1 - i + 2j + 1.5k), A_s a 14x17-grid 5-point reservoir operator (log-normal "
                               "permeability, upwind drift) standing in for saylr1; B uniform, m = 3..12 columns; "
                               "unrestarted Gl-QFOM / Gl-QGMRES, plain and QSAI-preconditioned (2 iterations)",
                   "l2": "the Krylov basis (at most 3000 x 0.27 MB) streams from HBM; no flush"},
        "e2e": {"value": 1e3 / e2e[0], "unit": "solves/s", "h2d_bytes_per_step": e2e[1], "d2h_bytes_per_step": e2e[2]},
        "gpu_launches": launches, "roofline": roof, "cpu_baseline": base, "result": out,
        "clocks": clk.summary()}), flush=True)
    return 0


def bench_learned(args, torch, qpinv):
    """Learned initial scaling: train the MLP on generator families at sizes
    32..256, then solve held-out full-rank 1024^2 and 2048 x 1024 matrices
    (log-uniform / geometric / clustered spectra, kappa <= 1e5) with the safe
    and the learned alpha (MIXED), and one with the plain FP64 form."""
    import numpy as np

    from paper_2605_01464_gb300 import learned_alpha as LA

    def cuda(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()

    ctx = qpinv.Context(0)
    t0 = time.perf_counter()
    feats, labels, _ = LA.make_dataset_gpu(ctx, torch, args.train_count, 32, 512, seed=11)
    t_data = time.perf_counter() - t0
    t0 = time.perf_counter()
    loss = ctx.alpha_train(feats, labels, epochs=300, batch=100, lr=3e-3, seed=5)
    torch.cuda.synchronize()
    t_train = time.perf_counter() - t0
    rows = []
    shapes = [(1024, 1024), (2048, 1024), (2048, 2048), (4096, 4096), (4096, 2048)]
    with ClockSampler(0) as clk:
        for k, fam in enumerate(("logspaced", "geometric", "clustered")):
            for (m, n) in shapes:
                A = cuda(LA.heldout_matrix(fam, m, n, 700 + 10 * k + m // 1024 + n // 512, device="cuda")[0])
                res = {}
                for mode in ("safe", "learned"):
                    ctx.configure(alpha=mode)
                    _timed_solve(ctx, torch, A, "qhpi19", args.tol)  # warm-up
                    ms, info = _timed_solve(ctx, torch, A, "qhpi19", args.tol)
                    res[mode] = {"ms": ms, "iters": info["iters"], "E1_rel": info["E_rel"][0],
                                 "alpha_source": info["alpha_source"], "precision": info["precision"]}
                rows.append({"family": fam, "m": m, "n": n, **res})
        ctx.configure(alpha="safe")
        A = cuda(LA.heldout_matrix("logspaced", 1024, 1024, 700, device="cuda")[0])
        ctx.configure(precision="fp64")
        ms64, info64 = _timed_solve(ctx, torch, A, "qhpi19", args.tol)
        ctx.configure(precision="mixed", alpha="learned")
        msl, infol = _timed_solve(ctx, torch, A, "qhpi19", args.tol)
        ctx.configure(alpha="safe")
    # equal accuracy: rows where both solves reach the stated tolerance
    eq = [r for r in rows if r["safe"]["E1_rel"] <= 1e-10 and r["learned"]["E1_rel"] <= 1e-10]
    safe_ms = sum(r["safe"]["ms"] for r in eq)
    learned_ms = sum(r["learned"]["ms"] for r in eq)
    print(json.dumps({
        "metric": "held-out solve time, safe alpha / learned alpha (QHPI19, mixed, equal accuracy)",
        "value": safe_ms / learned_ms, "unit": "x", "n_gpus": 1, "steps": 1, "warmup": 1,
        "higher_is_better": True, "dtype": "bf16-split/f32-acc + exact-slice f64", "data": "synthetic",
        "config": {"workload": "MLP 32-64-64-1 trained on %d generator-family matrices (32..512, drawn on the GPU "
                               "in groups of one shape); held-out 1024^2, 2048x1024, 2048^2, 4096^2, 4096x2048 with "
                               "log-uniform / geometric / clustered spectra, kappa = 10^U[1,5]" % args.train_count},
        "training": {"samples": args.train_count, "final_loss": loss, "data_s": t_data, "train_s": t_train},
        "iters": {"safe": sum(r["safe"]["iters"] for r in rows), "learned": sum(r["learned"]["iters"] for r in rows)},
        "equal_accuracy_rows": len(eq), "rows_total": len(rows),
        "rows": rows,
        "vs_fp64_fixed_alpha": {"matrix": "logspaced 1024^2 (seed 700)", "fp64_safe_ms": ms64,
                                "fp64_E1_rel": info64["E_rel"][0], "mixed_learned_ms": msl,
                                "mixed_learned_E1_rel": infol["E_rel"][0], "speedup": ms64 / msl},
        "clocks": clk.summary()}), flush=True)
    return 0


# DRAM bytes (read + write) per issued tensor flop from one ncu capture of
# the current exact-slice kernel on an 8-slice 2048^3 product
# (profiles/k_qgemm_emu_2048_slices8.md: 4.28 GB for 18 passes); a launch's
# traffic is estimated as this times its issued flops.  None where no
# capture matches the launches the solve makes (the split GEMM's launches
# carry the fused combine epilogue, the captured one a plain store).
TRAFFIC_PER_ISSUED_FLOP = {"k_qgemm_emu": 4.28e9 / (18 * 32 * 2048.0 ** 3),
                           "k_qgemm_tc": None}


def kernel_rooflines(st):
    """Roofline entries of the two tensor-core GEMM kernels, dominant (by
    time) first: achieved = algorithmic flops per launch (32 per quaternion
    multiply-add) / average CUDA-event duration of a launch; issued = tensor
    flops actually executed (slice or split passes)."""
    bf16_burst, bf16_sust, hbm, src = peaks()
    out = []
    for key, name, desc in (("emu", "k_qgemm_emu", "fused exact-slice FP64-accurate quaternion GEMM"),
                            ("tc", "k_qgemm_tc", "BF16-split quaternion GEMM")):
        n = st["%s_gemm_launches" % key]
        t = st["%s_gemm_ms" % key]
        if n == 0 or t <= 0:
            continue
        ms = t / n
        alg = st["%s_gemm_flops" % key] / n / (ms * 1e-3) / 1e12
        iss = st["%s_gemm_flops_issued" % key] / n / (ms * 1e-3) / 1e12
        tpf = TRAFFIC_PER_ISSUED_FLOP[name]
        traffic = tpf * st["%s_gemm_flops_issued" % key] / n if tpf else None
        out.append({"bound": "tensor", "achieved": alg, "peak": bf16_sust, "unit": "TFLOP/s",
                    "frac": alg / bf16_sust, "traffic": traffic, "traffic_unit": "bytes per launch (estimate)",
                    "kernel": "%s (%s)" % (name, desc), "launches": n, "ms_per_launch": ms, "total_ms": t,
                    "achieved_issued": iss, "frac_issued": iss / bf16_sust,
                    "peak_source": "%s bf16_tflops_sustained (MEASURED_PEAKS.json)" % src})
    out.sort(key=lambda r: -r["total_ms"])
    # the HBM-bound passes that remain outside the GEMM epilogues (FP64-master
    # combines, exact slicing, norms): bytes counted per launch by the library
    # (every plane read or written once), over their summed event time
    if st.get("ew_launches") and st.get("ew_ms", 0.0) > 0:
        gbs = st["ew_bytes"] / (st["ew_ms"] * 1e-3) / 1e9
        out.append({"bound": "hbm", "achieved": gbs, "peak": hbm, "unit": "GB/s", "frac": gbs / hbm,
                     "traffic": None, "kernel": "elementwise passes (combine, exact slicing, exponents, norms)",
                     "launches": st["ew_launches"], "total_ms": st["ew_ms"],
                     "ms_per_launch": st["ew_ms"] / st["ew_launches"],
                     "bytes_per_launch": st["ew_bytes"] / st["ew_launches"],
                     "peak_source": "%s hbm_gbs (MEASURED_PEAKS.json)" % src})
    return out or [None]


def reduce_timing(seconds, units, dist, device):
    """Replicas on N GPUs: the job's time is the slowest rank's, its work the
    sum of all ranks' units.  Returns (max seconds, total units); a no-op
    without a process group."""
    if dist is None:
        return seconds, units
    import torch
    t = torch.tensor([seconds], dtype=torch.float64, device=device)
    u = torch.tensor([float(units)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    dist.all_reduce(u, op=dist.ReduceOp.SUM)
    return float(t.item()), float(u.item())


def workload_config(args):
    return {"workload": "square %dx%d quaternion A = U diag(sigma) V^H, Haar U and V, sigma log-spaced 1..1e-6; "
                        "%s, mixed precision (BF16-split tensor-core products with FP32 accumulation; exact-slice "
                        "tensor-core X-products once ||A|| ||X|| > 1e3; %d polish iterations with FP64 masters and "
                        "FP64-accurate X-products), safe fixed alpha, rel. tol %g, FP64-accurate Penrose residuals" %
                        (args.n, args.n, args.method.upper(), args.polish, args.tol),
            "m": args.n, "n": args.n, "method": args.method, "precision": "mixed",
            "l2": "inputs exceed L2 (A alone is 134 MB of FP64 planes; no flush)"}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--n", type=int, default=2048)
    ap.add_argument("--method", default="qhpi19", choices=["ns", "qsai", "qrapid", "qhpi19", "qhpim"])
    ap.add_argument("--tol", type=float, default=1e-12)
    ap.add_argument("--polish", type=int, default=2)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-gemm-records", action="store_true",
                    help="skip the single-pass GEMM records at n = 4096 and 8192 in the default line")
    ap.add_argument("--kernel", default=None, choices=["qgemm"],
                    help="time only the tensor-core quaternion GEMM (n x n x n) for kernel profiling")
    ap.add_argument("--split", type=int, default=1,
                    help="--kernel qgemm: BF16 terms (tc: 1..3) or exact slices (emu: 2..8)")
    ap.add_argument("--gemm-precision", default="tc", choices=["tc", "emu"], help="--kernel qgemm precision")
    ap.add_argument("--emu-pair", default="auto", choices=["auto", "0", "1"],
                    help="--kernel qgemm: accepted, without effect (one exact-slice kernel serves every size)")
    ap.add_argument("--workload", default="dense",
                    choices=["dense", "batched", "rankdef", "learned", "hyper", "cur", "filter", "krylov"],
                    help="dense: one 2048^2 solve per step; batched: 4096 pure-quaternion blocks per step; "
                         "rankdef: rank-2048 8192x4096 (QHPI19 and NS, EMU); learned: learned-alpha training "
                         "and held-out evaluation; hyper: factorized vs unfactorized hyperpower (Example 3); "
                         "cur: CUR image completion (Sec. 5.1); filter: Lorenz signal filtering (Sec. 5.2); "
                         "krylov: QSAI-preconditioned global Krylov solvers (Sec. 3.5)")
    ap.add_argument("--train-count", type=int, default=20000, help="--workload learned: training matrices")
    ap.add_argument("--batch-count", type=int, default=4096,
                    help="--workload batched: blocks per step (4096 is the workload; fewer only for profiling)")
    ap.add_argument("--gen-device", default="cuda", choices=["cuda", "cpu"],
                    help="device that builds the synthetic input (cpu under profilers)")
    args = ap.parse_args()

    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if args.impl == "reference":
        return run_reference(args, rank)

    import numpy as np
    import torch

    from paper_2605_01464_gb300 import build as libbuild
    from paper_2605_01464_gb300 import qpinv

    libbuild.build()
    torch.cuda.set_device(local)
    if args.kernel == "qgemm":
        return kernel_qgemm(args, torch, qpinv)
    if args.workload == "batched":
        return bench_batched(args, torch, qpinv, world, rank, local)
    if args.workload == "rankdef":
        return bench_rankdef(args, torch, qpinv)
    if args.workload == "learned":
        return bench_learned(args, torch, qpinv)
    if args.workload == "hyper":
        return bench_hyper(args, torch, qpinv)
    if args.workload == "cur":
        return bench_cur(args, torch, qpinv)
    if args.workload == "filter":
        return bench_filter(args, torch, qpinv)
    if args.workload == "krylov":
        return bench_krylov(args, torch, qpinv)
    dist = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))

    A_host, U_host, s_host, V_host = make_workload(args.n, "cuda:%d" % local if args.gen_device == "cuda" else "cpu")
    A = torch.from_numpy(A_host).cuda()
    stream = torch.cuda.current_stream()
    ctx = qpinv.Context(local, precision="mixed", polish_iters=args.polish, profile=True)
    for _ in range(args.warmup):
        X, info = ctx.solve(A, args.method, tol=args.tol, max_iter=200, stream=stream)
    torch.cuda.synchronize()
    if dist:
        dist.barrier()
    ctx.reset_stats()
    ev0, ev1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    infos = []
    with ClockSampler(local) as clk:
        torch.cuda.synchronize()
        ev0.record(stream)
        for _ in range(args.steps):
            X, info = ctx.solve(A, args.method, tol=args.tol, max_iter=200, stream=stream)
            infos.append(info)
        ev1.record(stream)
        torch.cuda.synchronize()
    ms = ev0.elapsed_time(ev1)
    st = ctx.stats()
    sec, units = reduce_timing(ms / 1e3, args.steps, dist, "cuda")
    ms = sec * 1e3
    value = units / sec

    # end to end: host (pinned) A in, host X out, through the same C-ABI call
    e2e = None
    if not args.no_e2e:
        Ah = torch.from_numpy(A_host).pin_memory()
        Xh = torch.empty((4, args.n, args.n), dtype=torch.float64).pin_memory()
        ctx.configure(profile=False)
        ctx.solve(Ah, args.method, tol=args.tol, max_iter=200, X=Xh, stream=stream)
        torch.cuda.synchronize()
        if dist:
            dist.barrier()
        t0 = time.perf_counter()
        for _ in range(args.steps):
            _, info_h = ctx.solve(Ah, args.method, tol=args.tol, max_iter=200, X=Xh, stream=stream)
        torch.cuda.synchronize()
        te, units = reduce_timing(time.perf_counter() - t0, args.steps, dist, "cuda")
        nbytes = 4 * args.n * args.n * 8
        e2e = {"value": units / te, "unit": "solves/s", "h2d_bytes_per_step": nbytes,
               "d2h_bytes_per_step": nbytes + 8 * 4 * 3}

    if rank != 0:
        if dist:
            dist.destroy_process_group()
        return 0
    roofs = kernel_rooflines(st)
    if not args.no_gemm_records:
        roofs += gemm_target_records(torch, qpinv, local)
    last = infos[-1]
    line = {
        "metric": METRIC, "value": value, "unit": "solves/s", "n_gpus": world, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms / args.steps, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "bf16-split/f32-acc + exact-slice f64", "data": "synthetic",
        "config": workload_config(args),
        "roofline": roofs[0],
        "roofline_other": roofs[1:],
        "gpu_launches": st["kernel_launches"],
        "kernel_time_ms": {"emu_gemm": st["emu_gemm_ms"], "tc_gemm": st["tc_gemm_ms"], "f64_gemm": st["f64_gemm_ms"],
                           "elementwise": st["ew_ms"]},
        "result": {"iters": last["iters"], "tc_iters": last["tc_iters"], "polish_iters": last["polish_iters"],
                   "status": last["status"], "E_rel": last["E_rel"], "alpha": last["alpha"]},
        "clocks": clk.summary(),
        "e2e": e2e,
    }
    if world == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline_sample(A_host, last["iters"])
        err, secs = oracle_pinv_error(X.cpu().numpy(), U_host, s_host, V_host)
        line["result"]["x_relerr_vs_oracle"] = err
        line["result"]["x_relerr_reference"] = ("FP64 oracle V Sigma^-1 U^H of the generator's factors "
                                                "(%.1f s on the host cores)" % secs)
    print(json.dumps(line), flush=True)
    if dist:
        dist.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
