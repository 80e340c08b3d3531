"""Benchmark: regularized CCA solve (Alg. 1) to 1e-6 relative objective on the
tall BF16 workload (n = 262144, dx = dy = 512, k = 10, lambda = 1e-4, SRHT
s = 4096), one full solve per step (sketch + preconditioner + warm start +
Riemannian CG + FP64 Rayleigh-Ritz refinement), inputs resident in HBM.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Prints one JSON line (rank 0).  N > 1 runs N independent replicas (one per
GPU, launched by torch.distributed.run); value = whole-job time per solve.
"""
from __future__ import annotations

import argparse
import json
import os
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "CCA solve time to 1e-6 rel. objective; fused pass % of HBM peak; p50/p99 latency"
WORKLOAD = "cca_tall_bf16"
LAM = 1e-4
# Stopping rule.  The gradient rule ||grad||_M <= GTOL ||grad_0||_M is off:
# on this workload the CG gradient norm is not monotone and a threshold chosen
# on one instance stops other instances early.  The solve stops when the
# Rayleigh-Ritz values of span([U, eta]) (the values the final refinement
# reports) change by less than RTOL, relative, at two consecutive checks
# CHECK_EVERY iterations apart; tests/test_gpu_fullsize.py checks that this
# leaves every correlation within 1e-6 of the FP64 oracle on seeds 0, 1 and 2
# of the data and the sketch, and test_gpu_fp32_pass.py the same for FP32
# storage.
GTOL = 0.0
RTOL = 1e-7
CHECK_EVERY = 4
# Final Rayleigh-Ritz step from the Grams of the tensor-core pass (refine = 2;
# the same test checks this setting against the FP64 oracle).
REFINE = 2
# The LDA workload refines with FP64 Grams of W (refine = 1) and checks the
# Ritz values every 8 iterations (every 4 took more iterations to meet the
# rule on it: 161 against 137).
LDA_REFINE = 1
LDA_CHECK_EVERY = 8


# DRAM traffic of one full-size tc_pass_kernel launch (read + write bytes),
# from an ncu capture of 131072 rows of this workload (reads scaled by rows
# to 262144, partial writes as measured).  Valid only for the kernel source
# it was taken on (SHA-256 below); any other source reports null.
PASS_TRAFFIC_BYTES = 268.59008e6 * 2 + 9.76896e6
PASS_TRAFFIC_SRC_SHA256 = "15e3b8025cecca3cfe255afe45f453f04384e2b2294c55e31c554799c79abf92"


def pass_traffic():
    import hashlib
    path = os.path.join(ROOT, "paper_2106_12060_gb300", "csrc", "pass_tc.cu")
    try:
        with open(path, "rb") as f:
            h = hashlib.sha256(f.read()).hexdigest()
    except OSError:
        return None
    return PASS_TRAFFIC_BYTES if h == PASS_TRAFFIC_SRC_SHA256 else None


def peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            m = json.load(f)
        return float(m["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi samples of SM clock and throttle reasons while running."""

    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.index = index
        self.proc = None
        self.lines = []

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            self.lines.append(line.strip())

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        sm, smax, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for ln in self.lines:
            parts = [p.strip() for p in ln.split(",")]
            if len(parts) < 8:
                continue
            try:
                sm.append(float(parts[0]))
                smax.append(float(parts[1]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[4:8]):
                if val.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": float(np.median(sm)) if sm else None,
                "sm_max_mhz": float(max(smax)) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def dist_setup(args):
    import torch
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    if torch.cuda.is_available():
        torch.cuda.set_device(local)
    return ws, rank, local


def barrier(ws):
    if ws > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(ws, x: float) -> float:
    if ws == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([x], dtype=torch.float64, device="cuda" if torch.cuda.is_available() else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def workload_config(c, ws):
    """The `config` object of both arms' JSON lines."""
    return {"workload": WORKLOAD, "n": c["n"], "dx": c["dx"], "dy": c["dy"], "k": c["k"], "lambda": LAM,
            "sketch": "srht", "s": c["s"], "storage": c["dtype"], "gtol": GTOL, "rtol": RTOL,
            "check_every": CHECK_EVERY, "refine": REFINE,
            "parallelism": f"replicas{ws}", "l2": "inputs larger than L2 (537 MB)"}


def _threads():
    cores = len(os.sched_getaffinity(0)) if hasattr(os, "sched_getaffinity") else os.cpu_count()
    blas = None
    try:
        from threadpoolctl import threadpool_info
        blas = max([i.get("num_threads", 1) for i in threadpool_info()] or [1])
    except Exception:
        for var in ("OPENBLAS_NUM_THREADS", "OMP_NUM_THREADS", "MKL_NUM_THREADS"):
            if os.environ.get(var):
                blas = int(os.environ[var])
                break
    return cores, blas


def cpu_baseline(P, reps: int = 3):
    """The FP64 oracle timed at the FULL workload size on the host cores:
    route 2 (oracle.cca.cca_whiten: explicit Sigma, Cholesky whitening, SVD;
    the route the method's definition states) best and median of `reps`
    runs, and route 1 (oracle.cca.cca_qr: Householder QR of [Z; sqrt(lambda)
    I], the accurate route) once.  Returns the record and route 1's
    (sigma, U, V), which the caller also uses as the accuracy reference."""
    from oracle.cca import cca_whiten, cca_qr
    cores, blas = _threads()
    k = P["config"]["k"]
    n = P["X64"].shape[0]
    t2 = []
    for _ in range(reps):
        t0 = time.perf_counter()
        cca_whiten(P["X64"], P["Y64"], LAM, LAM, k)
        t2.append(time.perf_counter() - t0)
    t0 = time.perf_counter()
    ref = cca_qr(P["X64"], P["Y64"], LAM, LAM, k)
    t1 = time.perf_counter() - t0
    rec = {"value": float(np.median(t2)) * 1e3, "unit": "ms", "cores": blas or cores, "host_cores": cores,
           "blas_threads": blas, "kind": "oracle",
           "sample": f"the full {n}-row workload (no extrapolation): oracle.cca.cca_whiten (FP64 NumPy, "
                     f"route 2) median of {reps} runs; route 1 (oracle.cca.cca_qr) timed once",
           "route2_whiten_ms": {"median": float(np.median(t2)) * 1e3, "best": float(np.min(t2)) * 1e3,
                                "runs": len(t2)},
           "route1_qr_ms": {"once": t1 * 1e3}}
    return rec, ref


def accuracy_report(P, sig, U, V, ref):
    """Error of the GPU result against the FP64 oracle (route 1): canonical
    correlations, relative objective gap, and the largest sines of the
    principal angles between the GPU and oracle subspaces of U and V in the
    Sxx / Syy inner products (Def. 4.1 constraints)."""
    from oracle.cca import default_mu
    sr, Ur, Vr = ref
    s = sig.cpu().numpy()
    U = U.cpu().numpy()
    V = V.cpu().numpy()
    mu = default_mu(len(s))
    X, Y = P["X64"], P["Y64"]

    def sines(A, B, Z, lam):
        # principal angles in the (Z^T Z + lam I) inner product, from the thin
        # products with the data (no d x d Gram needed)
        def orth(M):
            ZM = Z @ M
            G = ZM.T @ ZM + lam * (M.T @ M)
            L = np.linalg.cholesky(G)
            return M @ np.linalg.inv(L).T
        Qa, Qb = orth(A), orth(B)
        C = (Z @ Qa).T @ (Z @ Qb) + lam * (Qa.T @ Qb)
        c = np.linalg.svd(C, compute_uv=False)
        return float(np.sqrt(max(0.0, 1.0 - min(1.0, float(np.min(c))) ** 2)))

    return {"sigma_max_rel_err": float(np.max(np.abs(s - sr) / sr)),
            "objective_rel_gap": float(abs(np.dot(mu, sr) - np.dot(mu, s)) / np.dot(mu, sr)),
            "subspace_sin_U": sines(U, Ur, X, LAM), "subspace_sin_V": sines(V, Vr, Y, LAM),
            "reference": "oracle.cca.cca_qr (FP64, route 1) on the stored BF16 values"}


def quantization_gap(P):
    """The canonical correlations of the stored BF16 values against those of
    the FP32 values they were rounded from (oracle route 2 on both): how much
    BF16 storage changes the problem itself, apart from any solver error."""
    from oracle.cca import cca_whiten
    from synth import make_workload
    Q = make_workload("cca_tall_f32", seed=P["config"]["seed"])
    k = P["config"]["k"]
    s16 = cca_whiten(P["X64"], P["Y64"], LAM, LAM, k)[0]
    s32 = cca_whiten(Q["X64"], Q["Y64"], LAM, LAM, k)[0]
    return {"sigma_max_rel_diff_bf16_vs_f32_data": float(np.max(np.abs(s16 - s32) / s32)),
            "sigma_f32_data": [float(x) for x in s32], "sigma_bf16_data": [float(x) for x in s16]}


def fp64_comparison(gb, P, sig_bf16, steps: int = 2):
    """The same solve (same sketch draws, stopping rule and refinement) with
    the data stored in FP64 (the BF16 values, exactly: the same problem) and
    the FP64 CUDA-core pass: the plain FP64 form on the same GPU."""
    import torch
    c = P["config"]
    n, dx, dy, k = c["n"], c["dx"], c["dy"], c["k"]
    X = torch.from_numpy(np.ascontiguousarray(P["X64"])).cuda()
    Y = torch.from_numpy(np.ascontiguousarray(P["Y64"])).cuda()
    opt = gb.default_options(sketch=gb.SRHT, s=c["s"], seed=c["seed"], max_iter=1000, gtol=GTOL, rtol=RTOL,
                             check_every=CHECK_EVERY)
    plan = gb.cca_plan(n, dx, dy, k, "f64", opt)
    U = torch.empty(dx, k, dtype=torch.float64, device="cuda")
    V = torch.empty(dy, k, dtype=torch.float64, device="cuda")
    sig = torch.empty(k, dtype=torch.float64, device="cuda")
    stream = torch.cuda.current_stream()

    def step():
        gb.cca_precondition(plan, X, Y, LAM, LAM)
        return gb.cca_solve(plan, U=U, V=V, sigma=sig)[3]

    step()
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    infos = [step() for _ in range(steps)]
    e1.record(stream)
    torch.cuda.synchronize()
    ms = e0.elapsed_time(e1) / steps
    s64 = sig.cpu().numpy()
    s16 = sig_bf16.cpu().numpy()
    plan.close()
    del X, Y
    torch.cuda.empty_cache()
    return {"ms": ms, "steps": steps, "storage": "f64", "iterations": float(np.mean([i["iters"] for i in infos])),
            "passes_per_solve": float(np.mean([i["passes"] for i in infos])),
            "sigma_max_rel_diff_vs_bf16": float(np.max(np.abs(s64 - s16) / np.abs(s64)))}


def other_workloads(gb, steps: int = 2):
    """The FP32 forms of the hot path, each one full solve per step with the
    data kernels of every pass timed by CUDA events: the tall CCA workload
    stored in FP32 (CUDA-core CCA pass) and the Fisher LDA workload (n =
    100000, d = 784, 10 classes, FP32; CUDA-core LDA pass, Alg. 2)."""
    import torch
    from synth import make_workload
    hbm, _ = peaks()
    out = {}
    stream = torch.cuda.current_stream()

    def timed(step):
        step()
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        infos = [step() for _ in range(steps)]
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / steps, infos

    P = make_workload("cca_tall_f32")
    c = P["config"]
    n, dx, dy, k = c["n"], c["dx"], c["dy"], c["k"]
    X = torch.from_numpy(np.ascontiguousarray(P["X"])).cuda()
    Y = torch.from_numpy(np.ascontiguousarray(P["Y"])).cuda()
    del P
    opt = gb.default_options(sketch=gb.SRHT, s=c["s"], seed=c["seed"], max_iter=1000, gtol=GTOL, rtol=RTOL,
                             check_every=CHECK_EVERY,
                             time_passes=1, refine=REFINE)
    plan = gb.cca_plan(n, dx, dy, k, "f32", opt)

    def cca_step():
        gb.cca_precondition(plan, X, Y, LAM, LAM)
        return gb.cca_solve(plan)[3]

    ms, infos = timed(cca_step)
    pass_ms = float(np.mean([i["pass_ms"] for i in infos]))
    gbps = n * (dx + dy) * 4 / (pass_ms * 1e-3) / 1e9
    out["cca_tall_f32"] = {"solve_ms": ms, "iterations": float(np.mean([i["iters"] for i in infos])),
                           "pass_ms": pass_ms, "pass_GBps": gbps, "pass_frac_of_hbm": gbps / hbm,
                           "pass_algorithmic_bytes": n * (dx + dy) * 4, "status": infos[-1]["status"],
                           "kernels": "tc_pass_kernel over the row-interleaved BF16 hi/lo copy of the FP32 "
                                      "data (2n rows; the hi-row and lo-row products summed in the epilogue), "
                                      "FP32 accumulate"}
    plan.close()
    del X, Y
    torch.cuda.empty_cache()

    P = make_workload("lda_f32")
    c = P["config"]
    n, d, l, k = c["n"], c["d"], c["l"], c["k"]
    Xh = np.ascontiguousarray(P["X"])
    y = P["y"].astype(np.int32)
    # lambda = 1e-6 tr(S_w) / d, the LDA workload's regularization rule:
    # tr(S_w) = sum_i ||x_i||^2 - sum_c n_c ||m_c||^2 (input preparation)
    x64 = Xh.astype(np.float64)
    cnt = np.bincount(y, minlength=l).astype(np.float64)
    sums = np.zeros((l, d))
    np.add.at(sums, y, x64)
    trsw = float(np.sum(x64 * x64) - np.sum(sums * sums / cnt[:, None]))
    lam = 1e-6 * trsw / d
    del x64
    X = torch.from_numpy(Xh).cuda()
    yl = torch.from_numpy(y).cuda()
    # the same Ritz-value stopping rule as the CCA solves, with the exact
    # (FP64) Rayleigh-Ritz refinement (tests/test_gpu_fullsize.py checks the
    # generalized eigenvalues against the oracle)
    opt = gb.default_options(s=c["s"], max_iter=1000, gtol=0.0, rtol=RTOL, check_every=LDA_CHECK_EVERY,
                             time_passes=1, refine=LDA_REFINE)
    plan = gb.lda_plan(n, d, l, k, "f32", opt)

    def lda_step():
        return gb.lda_solve(plan, X, yl, lam)[2]

    ms, infos = timed(lda_step)
    pass_ms = float(np.mean([i["pass_ms"] for i in infos]))
    nbytes = n * d * 4
    gbps = nbytes / (pass_ms * 1e-3) / 1e9
    out["lda_f32"] = {"solve_ms": ms, "iterations": float(np.mean([i["iters"] for i in infos])),
                      "rtol": RTOL, "refine": LDA_REFINE, "status": infos[-1]["status"], "pass_ms": pass_ms,
                      "pass_GBps": gbps, "pass_frac_of_hbm": gbps / hbm, "pass_algorithmic_bytes": nbytes,
                      "kernels": "tc_pass_kernel in one-view 2-CTA clusters (tcgen05 + TMA over the row-interleaved "
                                 "BF16 hi/lo copy of the class-centred FP32 data, the view's column pairs split over "
                                 "the two CTAs): Xhat^T (Xhat Phi)"}
    plan.close()
    del X
    torch.cuda.empty_cache()

    # the plain FP64 parity workload (n = 2000, dx = 50, dy = 40, k = 5,
    # CountSketch s = 360, gtol 1e-10): launch- and latency-bound, so the
    # figure of interest is the time per iteration
    P = make_workload("cca_small_fp64")
    c = P["config"]
    X = torch.from_numpy(np.ascontiguousarray(P["X"])).cuda()
    Y = torch.from_numpy(np.ascontiguousarray(P["Y"])).cuda()
    opt = gb.default_options(sketch=gb.COUNTSKETCH, s=c["s"], seed=c["seed"], max_iter=6000, gtol=0.0,
                             rtol=1e-10, check_every=CHECK_EVERY)
    plan = gb.cca_plan(c["n"], c["dx"], c["dy"], c["k"], "f64", opt)

    def small_step():
        gb.cca_precondition(plan, X, Y, c["lam"], c["lam"])
        return gb.cca_solve(plan)[3]

    ms, infos = timed(small_step)
    it = float(np.mean([i["iters"] for i in infos]))
    info = infos[-1]
    # accuracy against the FP64 oracle, and the first iterate whose relative
    # objective gap |sum mu sigma + f_t| / sum mu sigma is <= 1e-10 (from the
    # solver's per-iteration log of f)
    from oracle.cca import cca_qr, default_mu
    ref = cca_qr(P["X64"], P["Y64"], c["lam"], c["lam"], c["k"])[0]
    sig = torch.empty(c["k"], dtype=torch.float64, device="cuda")
    sig, _, _, info = gb.cca_solve(plan, sigma=sig)
    hist = gb.query(plan, gb.Q_HISTORY).cpu().numpy().reshape(-1, 3)[: info["iters"] + 1]
    opt_val = float(np.dot(default_mu(c["k"]), ref))
    gap = np.abs(opt_val + hist[:, 0]) / opt_val
    hit = np.nonzero(gap <= 1e-10)[0]
    us_it = 1e3 * ms / max(it, 1.0)
    out["cca_small_fp64"] = {
        "solve_ms": ms, "iterations": it, "us_per_iteration": us_it, "rtol": 1e-10,
        "status": gb.STATUS_NAMES.get(info["status"], info["status"]), "stalled": bool(info["stalled"]),
        "converged": info["status"] == gb.OK,
        "grad_ratio_final": info["grad_norm"] / info["grad_norm0"] if info["grad_norm0"] > 0 else None,
        "sigma_max_rel_err": float(np.max(np.abs(sig.cpu().numpy() - ref) / ref)),
        "iterations_to_1e-10_objective_gap": int(hit[0]) if hit.size else None,
        "time_to_1e-10_objective_gap_ms": float(hit[0] * us_it / 1e3) if hit.size else None,
        "note": "run to 1e-10: the Rayleigh-Ritz values of span([U, eta]) change by less than 1e-10 at two "
                "consecutive checks 8 iterations apart"}
    plan.close()
    return out


def batched_workload(gb, count: int = 64, seed: int = 0):
    """The uneven batched mix: `count` BF16 CCA instances, n log-uniform in
    [1e4, 2e6], dx, dy uniform over {64, ..., 1024}, k uniform over {1, 5, 10,
    20} (synth.batch_mix), data drawn on the device, CountSketch s = 4 (dx +
    dy), lambda 1e-3.  All instances are solved as one batch (one persistent
    tensor-core launch per iteration for the instances it serves, the others
    on their own passes) and, for comparison, one after another."""
    import torch
    from synth.batch_mix import batch_mix, latent_views_device
    hbm, _ = peaks()
    shapes = batch_mix(count, seed=seed)
    opt = dict(max_iter=1000, gtol=0.0, rtol=RTOL, check_every=CHECK_EVERY, refine=REFINE)
    plans, data = [], []
    t0 = time.perf_counter()
    for i, (n, dx, dy, k) in enumerate(shapes):
        X, Y = latent_views_device(n, dx, dy, seed=1000 + i)
        plan = gb.cca_plan(n, dx, dy, k, "bf16", gb.default_options(**opt))
        gb.cca_precondition(plan, X, Y, 1e-3, 1e-3)
        plans.append(plan)
        data.append((X, Y))
    torch.cuda.synchronize()
    prep_s = time.perf_counter() - t0
    batch = gb.Batch(plans)
    res, rep = gb.batch_solve(batch)  # tunes the schedule, captures the graphs
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record()
    res, rep = gb.batch_solve(batch)
    e1.record()
    torch.cuda.synchronize()
    batch_ms = e0.elapsed_time(e1)
    # the same instances solved one after another
    e0.record()
    solo = [gb.cca_solve(p) for p in plans]
    e1.record()
    torch.cuda.synchronize()
    seq_ms = e0.elapsed_time(e1)
    bytes_i = [n * (dx + dy) * 2 for (n, dx, dy, k) in shapes]
    passes = [r[3]["passes"] for r in res]
    moved = float(sum(b * p for b, p in zip(bytes_i, passes)))
    diff = max(float(torch.max(torch.abs(r[0] - s[0]) / s[0]).item()) for r, s in zip(res, solo))
    served = list(range(len(shapes)))  # every shape of the mix (BF16, d <= 1024, 16-byte rows)
    gbps = rep["batched_pass_bytes"] / (rep["batched_pass_ms"] * 1e-3) / 1e9 if rep["batched_pass_ms"] > 0 else None
    out = {
        "instances": count, "seed": seed, "total_data_GB": sum(bytes_i) / 1e9,
        "batch_solve_ms": batch_ms, "sequential_solves_ms": seq_ms, "speedup_vs_sequential": seq_ms / batch_ms,
        "lockstep_iterations": rep["iterations"],
        "iterations_mean": float(np.mean([r[3]["iters"] for r in res])),
        "iterations_max": int(max(r[3]["iters"] for r in res)),
        "status_ok": int(sum(1 for r in res if r[3]["status"] == gb.OK)),
        "sigma_max_rel_diff_vs_sequential": diff,
        "aggregate_GBps_over_solve": moved / (batch_ms * 1e-3) / 1e9,
        "aggregate_frac_of_hbm": moved / (batch_ms * 1e-3) / 1e9 / hbm,
        "batched_launch": {"instances": rep["batched_plans"], "clusters": rep["clusters"],
                           "bytes": rep["batched_pass_bytes"], "ms": rep["batched_pass_ms"],
                           "GBps": gbps, "frac_of_hbm": gbps / hbm if gbps else None,
                           "expected_instances": len(served)},
        "prepare_s": prep_s,
        "note": "a batched launch of 2-CTA clusters serves the instances with dx, dy <= 512 and k <= 12, two "
                "launches of the two-sweep pass the others (they read the data twice); the bytes, each plan's data "
                "once, and time are those of all launches",
    }
    batch.close()
    for p in plans:
        p.close()
    del data
    torch.cuda.empty_cache()
    return out


def serving_workload(gb, count: int = 128, n_max: float = 1e6, seed: int = 0, budget_gib: int = 120):
    """The serving stream: `count` requests (synth.batch_mix.serving_mix: 70%
    CCA / 30% FDA, n log-uniform in [1e4, n_max], widths log-uniform in [64,
    1024], CCA data BF16 or FP32 half and half) arriving as a Poisson process
    at 0.8x the throughput measured with the first requests all queued at
    once; HBM budget `budget_gib` GiB.  Every request's data is a row range
    of a device-resident pool (a latent-factor pair for CCA, a class-structured
    matrix for FDA) that the server copies in at admission.  Latency = finish
    - arrival (server clock); p50 / p99 over the stream."""
    import torch
    from synth.batch_mix import serving_mix, latent_views_device, lda_views_device
    reqs = serving_mix(count, n_range=(1e4, n_max), seed=seed)
    nmax = max(r["n"] for r in reqs)
    Xp, Yp = latent_views_device(nmax, 1024, 1024, seed=seed + 1)
    Xp32, Yp32 = Xp.float(), Yp.float()
    Lp, yp = lda_views_device(nmax, 1024, 21, seed=seed + 2)
    rng = np.random.default_rng(seed + 3)
    opt = dict(max_iter=1000, gtol=0.0, rtol=RTOL, check_every=CHECK_EVERY, refine=REFINE)

    def submit(srv, r):
        off = int(rng.integers(0, nmax - r["n"] + 1))
        rows = slice(off, off + r["n"])
        if r["kind"] == "cca":
            X, Y = (Xp, Yp) if r["dtype"] == "bf16" else (Xp32, Yp32)
            return srv.submit_cca(X[rows, :r["dx"]], Y[rows, :r["dy"]], r["k"], 1e-3, 1e-3,
                                  gb.default_options(**opt))
        labels = (yp[rows] % r["l"]).to(torch.int32).contiguous()
        return srv.submit_lda(Lp[rows, :r["d"]], labels, r["l"], r["k"], 1e-2, gb.default_options(**opt))

    def run(order, arrivals):
        srv = gb.Server(gb.default_server_options(hbm_budget=budget_gib << 30))
        t0 = time.perf_counter()
        ids, when, done = {}, {}, {}
        i = 0
        while i < len(order) or len(done) < len(order):
            now = time.perf_counter() - t0
            while i < len(order) and arrivals[i] <= now:
                rid = submit(srv, reqs[order[i]])
                ids[rid] = order[i]
                when[rid] = arrivals[i]
                i += 1
            q, r = srv.step()
            for rid in list(ids):
                if rid not in done and srv.state(rid) >= 2:
                    try:
                        vals, U, V, info, times = srv.result(rid)
                        done[rid] = (times["finish_s"] - when[rid], info["status"], info["iters"])
                    except gb.GbccaError as e:
                        done[rid] = (float("nan"), e.code, 0)
            if q == 0 and r == 0 and i < len(order):
                time.sleep(max(0.0, arrivals[i] - (time.perf_counter() - t0)))
        span = time.perf_counter() - t0
        srv.close()
        return done, span

    # saturated throughput: the first requests all queued at once
    m = min(32, count)
    sat, span = run(list(range(m)), [0.0] * m)
    rate = 0.8 * m / span
    gaps = rng.exponential(1.0 / rate, size=count)
    arrivals = np.cumsum(gaps) - gaps[0]
    done, span = run(list(range(count)), list(arrivals))
    lat = np.array([v[0] for v in done.values()])
    ok = [v for v in done.values() if v[1] == gb.OK]
    out = {
        "requests": count, "n_range": [1e4, n_max], "budget_GiB": budget_gib, "seed": seed,
        "saturated_solves_per_s": rate / 0.8,
        "arrival_rate_per_s": rate, "span_s": span, "solves_per_s": count / span,
        "p50_ms": float(np.nanpercentile(lat, 50) * 1e3), "p99_ms": float(np.nanpercentile(lat, 99) * 1e3),
        "mean_ms": float(np.nanmean(lat) * 1e3), "ok": len(ok), "failed": count - len(ok),
        "failed_status": {gb.STATUS_NAMES.get(c, str(c)): sum(1 for v in done.values() if v[1] == c)
                          for c in sorted({v[1] for v in done.values() if v[1] != gb.OK})},
        "iterations_mean": float(np.mean([v[2] for v in ok])) if ok else None,
        "mix": {"cca_bf16": sum(1 for r in reqs if r["kind"] == "cca" and r["dtype"] == "bf16"),
                "cca_f32": sum(1 for r in reqs if r["kind"] == "cca" and r["dtype"] == "f32"),
                "lda_f32": sum(1 for r in reqs if r["kind"] == "lda")},
        "note": "latency from the Poisson arrival time to the server's finish time of the request (admission "
                "wait, copy-in, preconditioning, iterations, refinement)",
    }
    del Xp, Yp, Xp32, Yp32, Lp, yp
    torch.cuda.empty_cache()
    return out


def run_reference(args, ws, rank):
    """The oracle as it stands on the host cores: every step is one FP64
    solve of the FULL workload by route 2 (oracle.cca.cca_whiten), timed
    with a wall clock; no sampling, no extrapolation."""
    if rank != 0:
        return
    from oracle.cca import cca_whiten
    from synth import make_workload
    P = make_workload(WORKLOAD)
    c = P["config"]
    cores, blas = _threads()

    def step():
        cca_whiten(P["X64"], P["Y64"], LAM, LAM, c["k"])

    for _ in range(args.warmup):
        step()
    vals = []
    for _ in range(args.steps):
        t0 = time.perf_counter()
        step()
        vals.append((time.perf_counter() - t0) * 1e3)
    v = float(np.mean(vals))
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": "ms", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": v, "higher_is_better": False,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": workload_config(c, args.gpus),
            "p50_ms": float(np.percentile(vals, 50)), "p99_ms": float(np.percentile(vals, 99)),
            "cpu_baseline": {"kind": "oracle", "cores": blas or cores, "host_cores": cores, "blas_threads": blas,
                             "sample": f"one full {c['n']}-row solve per step by oracle.cca.cca_whiten "
                                       f"(FP64 NumPy, route 2: explicit Sigma, Cholesky whitening, SVD)",
                             "value": v, "unit": "ms"},
            "e2e": {"value": v, "unit": "ms", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def run_ours(args, ws, rank, local):
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2106_12060_gb300 as gb
    from synth import make_workload

    P = make_workload(WORKLOAD)
    c = P["config"]
    n, dx, dy, k = c["n"], c["dx"], c["dy"], c["k"]
    dt = c["dtype"]

    def host_tensor(a):
        if dt == "bf16":
            return torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).view(torch.bfloat16)
        return torch.from_numpy(np.ascontiguousarray(a))

    Xh = host_tensor(P["X"]).pin_memory()
    Yh = host_tensor(P["Y"]).pin_memory()
    X = Xh.cuda()
    Y = Yh.cuda()
    stream = torch.cuda.current_stream()
    opt = gb.default_options(sketch=gb.SRHT, s=c["s"], seed=c["seed"], max_iter=1000, gtol=GTOL, rtol=RTOL,
                             check_every=CHECK_EVERY, time_passes=1, refine=REFINE)
    plan = gb.cca_plan(n, dx, dy, k, dt, opt)
    U = torch.empty(dx, k, dtype=torch.float64, device="cuda")
    V = torch.empty(dy, k, dtype=torch.float64, device="cuda")
    sig = torch.empty(k, dtype=torch.float64, device="cuda")

    def step(Xd, Yd):
        gb.cca_precondition(plan, Xd, Yd, LAM, LAM)
        return gb.cca_solve(plan, U=U, V=V, sigma=sig)[3]

    for _ in range(args.warmup):
        step(X, Y)
    torch.cuda.synchronize()
    sampler = ClockSampler(local)
    sampler.start()
    time.sleep(0.3)
    barrier(ws)
    torch.cuda.synchronize()
    l0 = gb.launch_count()
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps + 1)]
    ev[0].record(stream)
    infos = []
    for i in range(args.steps):
        infos.append(step(X, Y))
        ev[i + 1].record(stream)
    torch.cuda.synchronize()
    launches = gb.launch_count() - l0
    barrier(ws)
    per_step = [ev[i].elapsed_time(ev[i + 1]) for i in range(args.steps)]
    total_ms = ev[0].elapsed_time(ev[-1])
    total_ms = max_over_ranks(ws, total_ms)
    # end to end through the public API: pinned host inputs -> device -> solve -> host results
    Uh = torch.empty(dx, k, dtype=torch.float64).pin_memory()
    Vh = torch.empty(dy, k, dtype=torch.float64).pin_memory()
    sh = torch.empty(k, dtype=torch.float64).pin_memory()
    Xe = torch.empty_like(X)
    Ye = torch.empty_like(Y)
    barrier(ws)
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for i in range(args.steps):
        Xe.copy_(Xh, non_blocking=True)
        Ye.copy_(Yh, non_blocking=True)
        step(Xe, Ye)
        Uh.copy_(U, non_blocking=True)
        Vh.copy_(V, non_blocking=True)
        sh.copy_(sig, non_blocking=True)
    e1.record(stream)
    torch.cuda.synchronize()
    e2e_ms = max_over_ranks(ws, e0.elapsed_time(e1))
    # the same solves with every kernel launched directly (no graph replay)
    gopt = gb.default_options(sketch=gb.SRHT, s=c["s"], seed=c["seed"], max_iter=1000, gtol=GTOL, rtol=RTOL,
                              check_every=CHECK_EVERY, time_passes=0, refine=REFINE, graphs=0)
    gplan = gb.cca_plan(n, dx, dy, k, dt, gopt)

    def gstep():
        gb.cca_precondition(gplan, X, Y, LAM, LAM)
        return gb.cca_solve(gplan, U=U, V=V, sigma=sig)[3]

    for _ in range(args.warmup):
        gstep()
    barrier(ws)
    torch.cuda.synchronize()
    g0 = torch.cuda.Event(enable_timing=True)
    g1 = torch.cuda.Event(enable_timing=True)
    g0.record(stream)
    ginfos = [gstep() for _ in range(args.steps)]
    g1.record(stream)
    torch.cuda.synchronize()
    direct_ms = max_over_ranks(ws, g0.elapsed_time(g1)) / args.steps
    gplan.close()
    # the data pass alone, back to back at the solve's final point: one event
    # pair around 20 launches (no event between launches), for comparison
    # with the per-launch events inside the solve
    Px = torch.empty(dx, 2 * k, dtype=torch.float64, device="cuda")
    Py = torch.empty(dy, 2 * k, dtype=torch.float64, device="cuda")
    Px[:, :k] = U
    Px[:, k:] = 0.1 * torch.roll(U, 1, dims=1)
    Py[:, :k] = V
    Py[:, k:] = 0.1 * torch.roll(V, 1, dims=1)
    for _ in range(3):
        gb.fused_pass(plan, Px, Py)
    b0 = torch.cuda.Event(enable_timing=True)
    b1 = torch.cuda.Event(enable_timing=True)
    nb2b = 20
    b0.record(stream)
    for _ in range(nb2b):
        gb.fused_pass(plan, Px, Py)
    b1.record(stream)
    torch.cuda.synchronize()
    b2b_ms = b0.elapsed_time(b1) / nb2b
    clocks = sampler.stop()
    fp64 = None if args.no_fp64_compare else fp64_comparison(gb, P, sig)
    others = None if args.no_other_workloads else other_workloads(gb)
    batched = None if args.no_batched else batched_workload(gb)
    serving = None if args.no_serving else serving_workload(gb)

    hbm, peak_src = peaks()
    elt = {"bf16": 2, "f32": 4, "f64": 8}[dt]
    pass_bytes = n * (dx + dy) * elt
    pass_ms = float(np.mean([i["pass_ms"] for i in infos]))
    achieved = pass_bytes / (pass_ms * 1e-3) / 1e9
    value = total_ms / (args.steps * ws)
    line = {
        "metric": METRIC, "value": value, "unit": "ms", "n_gpus": ws, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": False,
        "scaling": "weak", "vs_baseline": None, "dtype": dt, "data": "synthetic",
        "config": workload_config(c, ws),
        "p50_ms": float(np.percentile(per_step, 50)), "p99_ms": float(np.percentile(per_step, 99)),
        "iterations": float(np.mean([i["iters"] for i in infos])),
        "passes_per_solve": float(np.mean([i["passes"] for i in infos])),
        "fused_pass": {"ms": pass_ms, "GBps": achieved, "frac_of_hbm": achieved / hbm,
                       "back_to_back": {"ms": b2b_ms, "GBps": pass_bytes / (b2b_ms * 1e-3) / 1e9,
                                        "frac_of_hbm": pass_bytes / (b2b_ms * 1e-3) / 1e9 / hbm,
                                        "note": "gbcca_fused_pass called 20 times back to back, one event "
                                                "pair around all 20; each call also runs the reduction, "
                                                "the Gram kernel and two copies"}},
        "roofline": {"bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s",
                     "frac": achieved / hbm, "traffic": pass_traffic(), "peak_source": peak_src,
                     "kernel": "tc_pass_kernel: fused CCA data pass (X^T W, Y^T W with W = [X Phi_x, Y Phi_y])",
                     "algorithmic_bytes": pass_bytes},
        "e2e": {"value": e2e_ms / (args.steps * ws), "unit": "ms",
                "h2d_bytes_per_step": int(Xh.numel() * Xh.element_size() + Yh.numel() * Yh.element_size()),
                "d2h_bytes_per_step": int(8 * (dx * k + dy * k + k))},
        "gpu_launches": int(launches),
        "clocks": clocks,
        "direct_launches": {"ms_per_solve": direct_ms, "steps": args.steps,
                            "iterations": float(np.mean([i["iters"] for i in ginfos])),
                            "note": "same solves with every kernel launched directly; the headline replays each "
                                    "batch of iterations from a captured CUDA graph (the library default), with "
                                    "the events around every data pass recorded by the graph"},
    }
    if fp64 is not None:
        fp64["bf16_speedup"] = fp64["ms"] / value
        line["fp64_gpu"] = fp64
    if others is not None:
        line["other_workloads"] = others
    if batched is not None:
        line["batched_uneven_mix"] = batched
    if serving is not None:
        line["serving"] = serving
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        line["cpu_baseline"], ref = cpu_baseline(P)
        line["accuracy"] = accuracy_report(P, sig, U, V, ref)
        line["quantization_gap"] = quantization_gap(P)
    if rank == 0:
        print(json.dumps(line), flush=True)
    plan.close()


def run_pass_only(args):
    """Only the fused data pass, `--pass-only ROWS` rows of the workload, for
    profiler captures (prints nothing that counts as a bench value)."""
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2106_12060_gb300 as gb
    from synth import make_workload
    torch.cuda.set_device(0)
    P = make_workload(args.workload, n=args.pass_only)
    c = P["config"]
    if c["kind"] == "lda":
        return run_pass_only_lda(args, P)
    n, dx, dy, k, dt = c["n"], c["dx"], c["dy"], c["k"], c["dtype"]
    to = (lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).view(torch.bfloat16).cuda()) \
        if dt == "bf16" else (lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda())
    X, Y = to(P["X"]), to(P["Y"])
    plan = gb.cca_plan(n, dx, dy, k, dt, gb.default_options(sketch=gb.COUNTSKETCH, warm_start=0))
    gb.cca_precondition(plan, X, Y, LAM, LAM)
    rng = np.random.default_rng(0)
    Px = torch.from_numpy(rng.standard_normal((dx, 2 * k)) / np.sqrt(dx)).cuda()
    Py = torch.from_numpy(rng.standard_normal((dy, 2 * k)) / np.sqrt(dy)).cuda()
    for _ in range(args.steps):
        gb.fused_pass(plan, Px, Py)
    torch.cuda.synchronize()
    print(f"pass-only: {args.steps} passes over {n} rows done")
    plan.close()


def run_pass_only_lda(args, P):
    """The FDA data pass of the LDA workload on its first rows, for profiler
    captures (prints nothing that counts as a bench value)."""
    import torch
    import paper_2106_12060_gb300 as gb
    c = P["config"]
    n, d, l, k, dt = c["n"], c["d"], c["l"], c["k"], c["dtype"]
    X = torch.from_numpy(np.ascontiguousarray(P["X"])).cuda()
    y = torch.from_numpy(P["y"]).cuda()
    plan = gb.lda_plan(n, d, l, k, dt, gb.default_options(s=c["s"], max_iter=1))
    gb.lda_solve(plan, X, y, 1e-3)
    rng = np.random.default_rng(0)
    Phi = torch.from_numpy(rng.standard_normal((d, 2 * k)) / np.sqrt(d)).cuda()
    for _ in range(args.steps):
        gb.fused_pass(plan, Phi)
    torch.cuda.synchronize()
    print(f"pass-only: {args.steps} FDA passes over {n} rows done")
    plan.close()


def run_solve_only(args):
    """Full solves (bench settings) on the first `--solve-rows ROWS` rows of
    the workload, for profiler captures of the per-iteration kernels (prints
    nothing that counts as a bench value)."""
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2106_12060_gb300 as gb
    from synth import make_workload
    torch.cuda.set_device(0)
    P = make_workload(args.workload, n=args.solve_rows)
    c = P["config"]
    n, dx, dy, k, dt = c["n"], c["dx"], c["dy"], c["k"], c["dtype"]
    to = (lambda a: torch.from_numpy(np.ascontiguousarray(a).view(np.int16)).view(torch.bfloat16).cuda()) \
        if dt == "bf16" else (lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda())
    X, Y = to(P["X"]), to(P["Y"])
    opt = gb.default_options(sketch=gb.SRHT, s=c["s"], seed=c["seed"], max_iter=1000, gtol=GTOL, rtol=RTOL,
                             check_every=CHECK_EVERY, refine=REFINE)
    plan = gb.cca_plan(n, dx, dy, k, dt, opt)
    for _ in range(args.steps):
        gb.cca_precondition(plan, X, Y, LAM, LAM)
        info = gb.cca_solve(plan)[3]
    torch.cuda.synchronize()
    print(f"solve-only: {args.steps} solves over {n} rows, {info['iters']} iterations")
    plan.close()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-fp64-compare", action="store_true",
                    help="skip the timed solve of the same workload stored in FP64")
    ap.add_argument("--no-other-workloads", action="store_true",
                    help="skip the FP32 CCA and FP32 LDA solves")
    ap.add_argument("--no-batched", action="store_true", help="skip the batched uneven-mix workload")
    ap.add_argument("--batched-only", action="store_true", help=argparse.SUPPRESS)
    ap.add_argument("--no-serving", action="store_true", help="skip the serving stream")
    ap.add_argument("--serving-only", action="store_true", help=argparse.SUPPRESS)
    ap.add_argument("--pass-only", type=int, default=0, help=argparse.SUPPRESS)
    ap.add_argument("--solve-rows", type=int, default=0, help=argparse.SUPPRESS)
    ap.add_argument("--workload", default=WORKLOAD, help=argparse.SUPPRESS)
    args = ap.parse_args()
    if args.pass_only:
        run_pass_only(args)
        return
    if args.solve_rows:
        run_solve_only(args)
        return
    if args.batched_only:
        import torch
        import __graft_entry__ as g
        g.build()
        import paper_2106_12060_gb300 as gb
        torch.cuda.set_device(0)
        print(json.dumps({"batched_uneven_mix": batched_workload(gb)}), flush=True)
        return
    if args.serving_only:
        import torch
        import __graft_entry__ as g
        g.build()
        import paper_2106_12060_gb300 as gb
        torch.cuda.set_device(0)
        print(json.dumps({"serving": serving_workload(gb)}), flush=True)
        return
    ws, rank, local = dist_setup(args)
    if args.impl == "reference":
        run_reference(args, ws, rank)
    else:
        run_ours(args, ws, rank, local)
    if ws > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
