"""Benchmark: SpMV sweep over CSR / ELL / SELL-P, FP64 and FP32, on the 3D
7-point Laplacian 256^3 and the Zipf(1.8) power-law matrix with 2^22 rows
(the paper's SpMV benchmark x = A b with random b, Section 6.1, on
synthetic stand-ins for its SuiteSparse set), plus CG solves/s on the 64x64
5-point Laplacian to a 1e-10 relative residual.

One step = one apply per (matrix, dtype) in the fastest of CSR / ELL /
SELL-P / COO for that matrix (picked by a short timing pass before the
timed region, as the paper reports each library's best-performing format,
Section 6).  value = algorithmic bytes of the step / device time (GB/s),
where every matrix counts its CSR algorithmic bytes = nnz*(value+index
bytes) + 4*(n+1) + x and y once, whichever format ran.  Every format is also
timed and listed under "sweep" with its own algorithmic bytes (ELL/SELL-P
unpadded without the row pointer, COO with a row index per entry).  The last
line on stdout is the result; the same with every section in full goes to
stderr.
Matrices (0.9-1.7 GB each) are larger than L2, so no flush is needed.
Extra keys: CG solves/s on the 64x64 Laplacian, time to 1e-10 on the 128^3
diffusion problem for FP32-refined vs plain FP64 Jacobi-CG / GMRES(30) /
CGS, the paper's fixed-1000-iteration time per iteration of CG, CGS and
GMRES(30), 2048 batched systems in one launch vs a per-system loop, and
serving latency.

python bench.py [--gpus N --steps K --warmup W] [--impl reference]
"""
from __future__ import annotations

import argparse
import hashlib
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

import numpy as np  # noqa: E402

METRIC = "SpMV GB/s & %HBM peak; CG solves/s at 1e-10 residual; serving p50/p99 latency"
WORKLOAD = ("SpMV, best of {CSR, ELL, SELL-P(S=32), COO} per matrix, {FP64, FP32}: 3D 7-point "
            "Laplacian 256^3 (n=16,777,216, nnz=117,047,296) and Zipf(1.8) power-law "
            "n=4,194,304 (mean 16, max 4096; ELL not built: ~206 GB padded); int32 indices; "
            "x ~ U[-1,1]")
FALLBACK_HBM = 6800.0


def _peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        with open(p) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    return FALLBACK_HBM, "fallback"


def job_throughput(local_ms, step_bytes, steps, world, device="cpu"):
    """Whole-job GB/s of `world` replicas that each ran `steps` steps of
    `step_bytes` algorithmic bytes: the job's time is the slowest rank's
    (an all_reduce MAX over the default process group when world > 1).
    Returns (job ms, GB/s)."""
    total_ms = float(local_ms)
    if world > 1:
        import torch
        import torch.distributed as dist
        t = torch.tensor([total_ms], dtype=torch.float64, device=device)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        total_ms = float(t.item())
    return total_ms, step_bytes * steps * world / (total_ms / 1000.0) / 1e9


def alg_bytes(m, sv, fmt):
    """Algorithmic bytes of one SpMV: unpadded matrix, x and y once."""
    b = m.nnz * (sv + 4) + m.n * sv + m.ncols * sv
    if fmt == "csr":
        b += 4 * (m.n + 1)
    if fmt == "coo":
        b += 4 * m.nnz  # the row index of every entry
    return int(b)


def build_items(gk, W, dtypes=("f64", "f32")):
    """Returns the sweep items (matrix handles + metadata)."""
    items = []
    lap = W.laplacian_3d(256)
    pl = W.power_law(1 << 22, seed=W.SEED_BASE + 2)
    for m, tag, fmts in ((lap, "lap3d_256", ("csr", "ell", "sellp", "coo")),
                         (pl, "powerlaw_4M", ("csr", "sellp", "coo"))):
        for dt in dtypes:
            sv = 8 if dt == "f64" else 4
            A = gk.Matrix.from_csr(m, dt)
            for fmt in fmts:
                H = A if fmt == "csr" else A.convert(fmt, None, 32, 1)
                items.append({"name": f"{tag}/{fmt}/{dt}", "mat": H, "dtype": dt, "fmt": fmt,
                              "n": m.n, "ncols": m.ncols, "nnz": m.nnz,
                              "bytes": alg_bytes(m, sv, fmt),
                              "csr_bytes": alg_bytes(m, sv, "csr"),
                              "kernel": H.desc["spmv_kernel"],
                              "launches": H.desc["spmv_launches"]})
    return items, lap, pl


KERNEL_NAMES = {0: "k_csr_vector", 1: "k_csr_rowtile", 2: "k_csr_seg", 3: "k_ell",
                4: "k_sellp", 5: "k_coo_warp", 6: "k_csr_warptile"}


class ClockSampler:
    """Samples nvidia-smi clocks and throttle reasons every 200 ms."""

    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, index=0):
        self.index = index
        self.samples = []
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--id={self.index}", f"--query-gpu={self.Q}",
                 "--format=csv,noheader,nounits", "-lms", "200"],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.thread = threading.Thread(target=self._read, daemon=True)
            self.thread.start()
        except Exception:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 7:
                self.samples.append(parts)

    def stop(self):
        if self.proc is not None:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except Exception:
                self.proc.kill()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        sm = [float(s[0]) for s in self.samples if s[0].replace(".", "").isdigit()]
        mx = [float(s[1]) for s in self.samples if s[1].replace(".", "").isdigit()]
        reasons = set()
        for s in self.samples:
            for i, nm in enumerate(names):
                if s[3 + i].lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(self.samples)}


def kernel_src_hash():
    h = hashlib.sha256()
    for f in ("spmv.cuh", "prims.cuh", "gk_internal.cuh", "apply.cu"):
        with open(os.path.join(ROOT, "paper_2510_08230_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    return h.hexdigest()[:16]


def traffic_for(kernel_name, item_name):
    """DRAM bytes per launch from a committed ncu capture, if the kernel
    sources are unchanged since it was taken."""
    p = os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(p):
        return None
    with open(p) as f:
        d = json.load(f)
    e = d.get(item_name)
    if not e or e.get("kernel") != kernel_name or e.get("src_hash") != kernel_src_hash():
        return None
    return e.get("dram_bytes_per_launch")


def cpu_baseline(lap, seconds=12.0):
    """The oracle's row-parallel FP64 CSR SpMV on the host cores, on the
    256^3 Laplacian, repeated for about `seconds`."""
    import oracle
    rp = np.ascontiguousarray(lap.row_ptr, dtype=np.int32)
    ci = np.ascontiguousarray(lap.col_idx, dtype=np.int32)
    va = np.ascontiguousarray(lap.values, dtype=np.float64)
    x = np.random.default_rng(1).uniform(-1, 1, lap.n)
    y = np.zeros(lap.n)
    oracle.spmv_omp(lap, x, 0, y=y, arrays=(rp, ci, va))  # warm-up
    reps, t0 = 0, time.perf_counter()
    threads = 0
    while True:
        _, threads = oracle.spmv_omp(lap, x, 0, y=y, arrays=(rp, ci, va))
        reps += 1
        el = time.perf_counter() - t0
        if el >= seconds or reps >= 5000:
            break
    gbs = alg_bytes(lap, 8, "csr") * reps / el / 1e9
    return {"value": round(gbs, 2), "unit": "GB/s", "cores": int(threads), "kind": "oracle",
            "sample": f"{reps} x FP64 CSR SpMV of the 3D 7-point 256^3 Laplacian (row-parallel "
                      f"OpenMP oracle, plain sum), {el:.1f} s"}


def _x_err(x, xo):
    d = float(np.linalg.norm(xo))
    return float(np.linalg.norm(np.asarray(x, np.float64) - xo) / d) if d > 0 else None


def oracle_legs(W, lap, keep, budget_s=60.0):
    """The CPU oracle beside the GPU results (rank 0, one replica only):
    - SpMV of the 256^3 Laplacian on one host thread (the OpenMP timing is
      cpu_baseline);
    - CG, BiCGSTAB and GMRES(30) to 1e-10 on the 64x64 Laplacian (no
      preconditioner, run to the end) and with Jacobi on the 128^3 diffusion
      matrix (CG run to the end; BiCGSTAB and GMRES(30) timed over a bounded
      number of iterations and extrapolated to the iteration count the GPU's
      FP64 solve needed);
    - a loop of oracle Jacobi-CG solves over the first batched systems for
      a bounded time, extrapolated to all 2048 by rows;
    - for every GPU solution kept by the solver legs: the true relative
      residual ||b - A x|| / ||b|| recomputed with the oracle's compensated
      SpMV, and ||x - x_oracle|| / ||x_oracle|| against the oracle's own
      solution of the same system (Jacobi-CG to 1e-10)."""
    import oracle
    t_start = time.perf_counter()
    out = {"kind": "oracle", "cores_spmv_single": 1}
    # single-thread SpMV
    rp = np.ascontiguousarray(lap.row_ptr, dtype=np.int32)
    ci = np.ascontiguousarray(lap.col_idx, dtype=np.int32)
    va = np.ascontiguousarray(lap.values, dtype=np.float64)
    xv = np.random.default_rng(1).uniform(-1, 1, lap.n)
    yv = np.zeros(lap.n)
    reps, t0 = 0, time.perf_counter()
    while True:
        oracle.spmv_omp(lap, xv, 1, y=yv, arrays=(rp, ci, va))
        reps += 1
        el = time.perf_counter() - t0
        if el >= 4.0:
            break
    out["spmv_single_thread"] = {
        "GB_s": round(alg_bytes(lap, 8, "csr") * reps / el / 1e9, 2), "reps": reps,
        "s": round(el, 2), "workload": "FP64 CSR SpMV of the 3D 7-point 256^3 Laplacian, 1 thread"}
    # config 1: the 64x64 Laplacian, no preconditioner
    m1 = W.laplacian_2d(64)
    b1 = W.uniform_vector(m1.n, W.SEED_BASE + 1)
    c1 = {}
    x1o = None
    for name, meth in (("cg", oracle.CG), ("bicgstab", oracle.BICGSTAB), ("gmres30", oracle.GMRES)):
        t0 = time.perf_counter()
        xo, io = oracle.solve(m1, b1, method=meth, tol=1e-10, max_iters=20000, krylov_dim=30)
        el = time.perf_counter() - t0
        c1[name] = {"ms": round(el * 1000, 3), "iters": io["iters"], "status": io["status"],
                    "rel_res_true": io["rel_res_true"], "solves_per_s": round(1.0 / el, 1)}
        if name == "cg":
            x1o = xo
    out["laplacian_64x64"] = c1
    # config 3: 128^3 diffusion with Jacobi
    m3 = W.diffusion_3d(128)
    b3 = W.uniform_vector(m3.n, W.SEED_BASE + 3)
    c3 = {}
    t0 = time.perf_counter()
    x3o, io = oracle.solve(m3, b3, method=oracle.CG, precond=1, tol=1e-10, max_iters=20000)
    el = time.perf_counter() - t0
    c3["cg_jacobi"] = {"s": round(el, 2), "iters": io["iters"], "status": io["status"],
                       "rel_res_true": io["rel_res_true"], "ms_per_iter": round(el * 1e3 / max(io["iters"], 1), 2),
                       "how": "run to the end"}
    for name, meth, gpu_key in (("bicgstab_jacobi", oracle.BICGSTAB, "ir_128cubed/bicgstab/fp64"),
                                ("gmres30_jacobi", oracle.GMRES, "ir_128cubed/gmres/fp64")):
        k = 30
        t0 = time.perf_counter()
        _, io = oracle.solve(m3, b3, method=meth, precond=1, tol=1e-10, max_iters=k, krylov_dim=30)
        el = time.perf_counter() - t0
        per = el / max(io["iters"], 1)
        gpu_iters = keep.get(gpu_key, (None, {}))[1].get("iters")
        c3[name] = {"ms_per_iter": round(per * 1e3, 2), "sample_iters": io["iters"],
                    "gpu_fp64_iters": gpu_iters,
                    "s_extrapolated": round(per * gpu_iters, 1) if gpu_iters else None,
                    "how": f"extrapolated: {io['iters']} oracle iterations timed, x the GPU "
                           "FP64 solve's iteration count"}
    out["diffusion_128cubed"] = c3
    # batched: oracle Jacobi-CG loop over the systems, bounded time
    mats, rhs = W.batched_rectangles(2048, seed=W.SEED_BASE + 4)
    xs_gpu = keep.get("batched_2048/f64")
    rows_done, done, errs, res = 0, 0, [], []
    t0 = time.perf_counter()
    for i, (m, b) in enumerate(zip(mats, rhs)):
        xo, io = oracle.solve(m, b, method=oracle.CG, precond=1, tol=1e-10, max_iters=20000)
        rows_done += m.n
        done += 1
        if xs_gpu is not None:
            errs.append(_x_err(xs_gpu[i], xo))
            res.append(oracle.true_rel_residual(m, b, xs_gpu[i]))
        if time.perf_counter() - t0 >= 12.0:
            break
    el = time.perf_counter() - t0
    total_rows = sum(m.n for m in mats)
    out["batched_2048"] = {
        "systems_timed": done, "s": round(el, 2),
        "s_extrapolated_all": round(el * total_rows / rows_done, 1),
        "how": "sequential oracle Jacobi-CG (FP64, 1e-10) loop over the first systems; "
               "extrapolated to all 2048 by rows",
        "gpu_batched_f64_max_rel_res_true_oracle": max(res) if res else None,
        "gpu_batched_f64_max_x_err_vs_oracle": max(errs) if errs else None,
        "systems_checked": len(errs)}
    # oracle error of every kept GPU solution
    checks = {}
    for key, val in keep.items():
        if key == "batched_2048/f64":
            continue
        x, rec = val
        if key.startswith("cg/"):
            m, b, xo = m1, b1, x1o
        else:
            m, b, xo = m3, b3, x3o
        checks[key] = {"rel_res_true_oracle": oracle.true_rel_residual(m, b, x),
                       "x_err_vs_oracle": _x_err(x, xo),
                       "gpu_rel_res_true": rec.get("rel_res_true")}
        rec["rel_res_true_oracle"] = checks[key]["rel_res_true_oracle"]
        rec["x_err_vs_oracle"] = checks[key]["x_err_vs_oracle"]
    out["gpu_results_vs_oracle"] = checks
    out["total_s"] = round(time.perf_counter() - t_start, 1)
    return out


def cg_solves_per_s(gk, W, torch, dev, reps=20, keep=None):
    m = W.laplacian_2d(64)
    b = torch.from_numpy(W.uniform_vector(m.n, W.SEED_BASE + 1)).to(dev)
    A = gk.Matrix.from_csr(m)
    x = torch.zeros_like(b)
    out = {}
    for engine in (1, 2, 3):
        A.solve(b, x, method="cg", tol=1e-10, max_iters=5000, engine=engine)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        iters = 0
        for _ in range(reps):
            x.zero_()
            info = A.solve(b, x, method="cg", tol=1e-10, max_iters=5000, engine=engine)
            assert info["return"] == gk.GK_OK, info
            iters = info["iters"]
        torch.cuda.synchronize()
        el = time.perf_counter() - t0
        tag = {1: "multi_kernel", 2: "single_block", 3: "cluster"}[engine]
        out[tag] = {"solves_per_s": round(reps / el, 1), "iters": iters,
                    "rel_res_true": info["rel_res_true"]}
        if keep is not None:
            keep[f"cg/{tag}"] = (x.cpu().numpy(), out[tag])
    A.close()
    best = max(out.values(), key=lambda v: v["solves_per_s"])
    return {"solves_per_s": best["solves_per_s"], "workload": "2D 5-point 64x64 FP64 CG to 1e-10, "
            "b ~ U[-1,1] seed 2511, x0 = 0 (host wall clock per solve incl. launch)",
            "engines": out}


def time_apply(it, stream, torch, reps=3):
    """Mean device time (ms) of `reps` applies of one sweep item."""
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    it["mat"].apply(it["x"], it["y"], stream)
    e0.record(stream)
    for _ in range(reps):
        it["mat"].apply(it["x"], it["y"], stream)
    e1.record(stream)
    torch.cuda.synchronize()
    return e0.elapsed_time(e1) / reps


def ir_compare(gk, W, torch, dev, keep=None):
    """128^3 log-normal diffusion: wall time to a true 1e-10 residual,
    FP32 inner solves in FP64 refinement vs plain FP64 (Jacobi-CG,
    Jacobi-GMRES(30) and Jacobi-CGS)."""
    m = W.diffusion_3d(128)
    b = torch.from_numpy(W.uniform_vector(m.n, W.SEED_BASE + 3)).to(dev)
    A = gk.Matrix.from_csr(m)
    out = {"workload": "128^3 7-point diffusion, exp(N(0,1)) cells, harmonic faces; "
                       "b ~ U[-1,1] seed 2513; x0 = 0; tol 1e-10 (true residual)"}
    for method in ("cg", "bicgstab", "gmres", "cgs"):
        res = {}
        for mixed in (0, 1, 2):
            x = torch.zeros_like(b)
            A.solve(b, x, method=method, precond="jacobi", tol=1e-10, max_iters=20000,
                    mixed=mixed)  # warm-up (plans, low-precision copy, graphs)
            x.zero_()
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            info = A.solve(b, x, method=method, precond="jacobi", tol=1e-10, max_iters=20000,
                           mixed=mixed)
            torch.cuda.synchronize()
            el = time.perf_counter() - t0
            tag = {0: "fp64", 1: "fp32_ir", 2: "bf16_ir"}[mixed]
            res[tag] = {
                "ms": round(el * 1000, 2), "status": info["return"], "iters": info["iters"],
                "outer": info["outer_iters"], "rel_res_true": info["rel_res_true"]}
            if keep is not None:
                keep[f"ir_128cubed/{method}/{tag}"] = (x.cpu().numpy(), res[tag])
        res["speedup_fp32_ir"] = round(res["fp64"]["ms"] / res["fp32_ir"]["ms"], 3)
        out[method] = res
    A.close()
    return out


def per_iteration_protocol(gk, W, torch, dev, iters=1000):
    """The paper's solver protocol (Section 6.2.1): a fixed 1000 iterations
    of CG, CGS and GMRES(30) without a preconditioner, reported as time per
    iteration, here on the 128^3 diffusion matrix (FP64).  A method that
    breaks down or reaches a residual of 1e-30 first is timed over the
    iterations it ran."""
    m = W.diffusion_3d(128)
    b = torch.from_numpy(W.uniform_vector(m.n, W.SEED_BASE + 3)).to(dev)
    A = gk.Matrix.from_csr(m)
    out = {"workload": "128^3 diffusion FP64, no preconditioner, 1000 iterations (GMRES: "
                       "Arnoldi steps, restart 30), x0 = 0; device time per iteration"}
    for method in ("cg", "cgs", "gmres"):
        x = torch.zeros_like(b)
        A.solve(b, x, method=method, tol=1e-30, max_iters=20)  # warm-up (graphs)
        x.zero_()
        torch.cuda.synchronize()
        info = A.solve(b, x, method=method, tol=1e-30, max_iters=iters, krylov_dim=30)
        its = max(int(info["iters"]), 1)
        out[method] = {"iters": int(info["iters"]), "status": info["return"],
                       "us_per_iter": round(info["device_ms"] * 1000.0 / its, 2),
                       "rel_res_true": info["rel_res_true"]}
    A.close()
    return out


def precond_compare(gk, W, torch, dev, keep=None):
    """CG and GMRES(30) to a true 1e-10 on the 128^3 diffusion matrix (FP64)
    without a preconditioner, with Jacobi, with block-Jacobi of 4, 8 and 16
    rows, and with ILU(0): iterations and wall time (host clock around the
    solve; the preconditioner is built by a warm-up solve first).  GMRES is
    capped at 5000 steps (status 1 if it had not converged).  Also the time
    of one ILU(0) application (both substitutions) in FP64 and FP32."""
    m = W.diffusion_3d(128)
    b = torch.from_numpy(W.uniform_vector(m.n, W.SEED_BASE + 3)).to(dev)
    A = gk.Matrix.from_csr(m)
    out = {"workload": "128^3 diffusion FP64, tol 1e-10, x0 = 0"}
    for method in ("cg", "gmres"):
        res = {}
        for label, kw in (("none", dict(precond=None)), ("jacobi", dict(precond="jacobi")),
                          ("block4", dict(precond="block_jacobi", block_size=4)),
                          ("block8", dict(precond="block_jacobi", block_size=8)),
                          ("block16", dict(precond="block_jacobi", block_size=16)),
                          ("ilu0", dict(precond="ilu"))):
            x = torch.zeros_like(b)
            A.solve(b, x, method=method, tol=1e-10, max_iters=20, **kw)  # warm-up (setup)
            x.zero_()
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            cap = 20000 if method == "cg" else 5000  # GMRES without M: bounded
            info = A.solve(b, x, method=method, tol=1e-10, max_iters=cap, **kw)
            torch.cuda.synchronize()
            res[label] = {"ms": round((time.perf_counter() - t0) * 1000, 2),
                          "iters": info["iters"], "status": info["return"],
                          "rel_res_true": info["rel_res_true"]}
            if keep is not None:
                keep[f"preconditioners/{method}/{label}"] = (x.cpu().numpy(), res[label])
        out[method] = res
    A.close()
    apply_us = {}
    for dt in ("f64", "f32"):
        vt = torch.float64 if dt == "f64" else torch.float32
        B = gk.Matrix.from_csr(m, dt)
        r = b.to(vt)
        z = torch.empty_like(r)
        B.precond_apply(r, z, "ilu")  # builds the factors
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        for _ in range(10):
            B.precond_apply(r, z, "ilu")
        torch.cuda.synchronize()
        apply_us[dt] = round((time.perf_counter() - t0) / 10 * 1e6, 1)
        B.close()
    out["ilu0_apply_us"] = apply_us
    return out


def abi_overhead(gk, W, torch, dev):
    """The paper's binding-overhead experiment (Section 6.3) for this
    library's ctypes binding: SpMV time through the Python binding against
    the native C driver (native/abi_overhead.c) on the same matrices, both
    timed per call on a host clock with a device synchronisation after each
    apply.  P_overhead = (P_native - P_python) / P_native * 100 with P in
    GFLOP/s (2 flops per nonzero); T_overhead = T_python - T_native."""
    import tempfile
    from paper_2510_08230_gb300 import _build
    exe = _build.build_native()
    out = {"workload": "2D 5-point Laplacians N x N, FP64, CSR and COO, x on the device; "
                       "per-call host clock after cudaDeviceSynchronize (paper Section 6.3)",
           "rows": []}
    for N in (16, 64, 256, 1024, 2048):
        m = W.laplacian_2d(N)
        reps = 2000 if m.nnz < 1e6 else 200
        with tempfile.NamedTemporaryFile(suffix=".csr", delete=False) as f:
            np.array([m.n, m.ncols], np.int32).tofile(f)
            np.array([m.nnz], np.int64).tofile(f)
            np.asarray(m.row_ptr, np.int32).tofile(f)
            np.asarray(m.col_idx, np.int32).tofile(f)
            np.asarray(m.values, np.float64).tofile(f)
            path = f.name
        try:
            for fmt in ("csr", "coo"):
                A = gk.Matrix.from_csr(m)
                if fmt == "coo":
                    B = A.convert("coo")
                    A.close()
                    A = B
                x = torch.zeros(m.n, dtype=torch.float64, device=dev)
                y = torch.empty_like(x)
                for _ in range(10):
                    A.apply(x, y)
                    torch.cuda.synchronize()
                t0 = time.perf_counter()
                for _ in range(reps):
                    A.apply(x, y)
                    torch.cuda.synchronize()
                t_py = (time.perf_counter() - t0) / reps
                A.close()
                r = subprocess.run([exe, path, fmt, str(reps)], capture_output=True, text=True,
                                   timeout=300)
                t_nat = float(r.stdout.strip()) if r.returncode == 0 else float("nan")
                flops = 2.0 * m.nnz
                p_py, p_nat = flops / t_py / 1e9, flops / t_nat / 1e9
                out["rows"].append({"N": N, "nnz": m.nnz, "format": fmt,
                                    "t_python_us": round(t_py * 1e6, 2),
                                    "t_native_us": round(t_nat * 1e6, 2),
                                    "T_overhead_us": round((t_py - t_nat) * 1e6, 2),
                                    "P_overhead_pct": round((p_nat - p_py) / p_nat * 100.0, 1)})
        finally:
            os.unlink(path)
    return out


def batched_compare(gk, W, torch, dev, count=2048, keep=None):
    """2048 shifted-rectangle SPD systems (64-4096 rows): one persistent
    launch vs a per-system gk_solve loop, CG to 1e-10, FP64 and FP32."""
    mats, rhs = W.batched_rectangles(count, seed=W.SEED_BASE + 4)
    out = {"workload": f"{count} 2D 5-point Laplacians on random rectangles + diagonal shift "
                       "U[0,1], n 64..4096, CG (Jacobi) to 1e-10 (FP64) / 1e-5 (FP32)"}
    for dt in ("f64", "f32"):
        vt = torch.float64 if dt == "f64" else torch.float32
        tol = 1e-10 if dt == "f64" else 1e-5
        As = [gk.Matrix.from_csr(m, dt) for m in mats]
        bs = [torch.from_numpy(b).to(dev, vt) for b in rhs]
        xs = [torch.zeros(m.n, dtype=vt, device=dev) for m in mats]
        opts = gk.make_opts(method="cg", precond="jacobi", tol=tol, max_iters=20000)
        gk.gk_solve_batched([A.handle for A in As], bs, xs, opts)  # warm-up
        for x in xs:
            x.zero_()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        st, infos = gk.gk_solve_batched([A.handle for A in As], bs, xs, opts)
        torch.cuda.synchronize()
        t_batch = time.perf_counter() - t0
        ok = sum(1 for i in infos if i["status"] == 0)
        names = {gk.GK_CSR: "csr", gk.GK_ELL: "ell", gk.GK_SELLP: "sellp"}
        chosen = {}
        for i in infos:
            k = (f"{names.get(i['spmv_format'], '?')}"
                 f"{i['slice_size'] if i['spmv_format'] == gk.GK_SELLP else ''}"
                 f"/{i['block_threads']}t")
            chosen[k] = chosen.get(k, 0) + 1
        if keep is not None and dt == "f64":
            keep["batched_2048/f64"] = [x.cpu().numpy() for x in xs]
        for x in xs:
            x.zero_()
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        loop_ok = 0
        for A, b, x in zip(As, bs, xs):
            info = A.solve(b, x, method="cg", precond="jacobi", tol=tol, max_iters=20000)
            loop_ok += info["return"] == 0
        torch.cuda.synchronize()
        t_loop = time.perf_counter() - t0
        out[dt] = {"batched_ms": round(t_batch * 1000, 2), "loop_ms": round(t_loop * 1000, 2),
                   "speedup": round(t_loop / t_batch, 2),
                   "solves_per_s_batched": round(count / t_batch, 1),
                   "autotuned_layouts": chosen,
                   "converged_batched": ok, "converged_loop": loop_ok}
        for A in As:
            A.close()
    return out


def serving_bench(gk, W, torch, dev, n_req=240, factors=((0.5, 400), (0.8, 2000), (0.95, 400)),
                  server_kw=None):
    """Config 5: Poisson arrivals of solve requests (2D/3D stencils and
    banded SPD, n log-uniform 1e3..1e6, FP64 or FP32-refined 50/50, tol
    log-uniform 1e-10..1e-8) under a 40 GB budget.  Saturation throughput is
    measured with a burst of n_req requests; then (rate factor, count)
    requests arrive at 0.5 / 0.8 / 0.95 x saturation (2000 at 0.8, so that
    its p99 rests on 20 samples).  Latency = submit -> x back on the host."""
    import threading
    from paper_2510_08230_gb300.serve import SolveRequest, SolveServer
    pool = W.serving_pool(24)
    rng = np.random.default_rng(W.SEED_BASE + 5)
    params = W.serving_requests(pool, n_req + sum(c for _, c in factors))
    rhs = {}

    def make(rid):
        mi, prec, tol, seed = params[rid]
        key = (mi, seed % 4)
        if key not in rhs:
            rhs[key] = W.uniform_vector(pool[mi].n, seed % 4 + 17 * mi)
        return SolveRequest(rid, mi, pool[mi], rhs[key], tol=tol, precision=prec)

    reqs = [make(i) for i in range(len(params))]
    srv = SolveServer(budget_bytes=40e9, **(server_kw or dict(workers=6)))
    # warm-up: every pool matrix once per precision (uploads, plans, graphs)
    warm = []
    for mi, m in enumerate(pool):
        for prec in ("f64", "ir32"):
            warm.append(srv.submit(SolveRequest(-1, mi, m, W.uniform_vector(m.n, 1), 1e-8, prec)))
    for r in warm:
        r.event.wait(600)
    out = {"workload": "24-matrix pool (2D 5-pt / 3D 7-pt / banded SPD w 5..64, n log-uniform "
                       "1e3..1e6), FP64 or FP32-refined 50/50, tol 1e-10..1e-8, Jacobi-CG, "
                       "40 GB budget, 6 workers (arrival order; small FP64 systems batched; "
                       "one stream priority), "
                       f"{n_req}-request burst, " +
                       ", ".join(f"{c} requests at {f}x" for f, c in factors)}
    burst = reqs[:n_req]
    t0 = time.perf_counter()
    for r in burst:
        srv.submit(r)
    for r in burst:
        r.event.wait(600)
    t1 = time.perf_counter()
    sat = n_req / (t1 - t0)
    out["saturation"] = SolveServer.summarize(burst, t0, t1)
    start = n_req
    for f, cnt in factors:
        batch = reqs[start:start + cnt]
        start += cnt
        gaps = rng.exponential(1.0 / (f * sat), size=len(batch))
        arrive = np.cumsum(gaps)

        def feeder():
            base = time.perf_counter()
            for r, a in zip(batch, arrive):
                dt = base + a - time.perf_counter()
                if dt > 0:
                    time.sleep(dt)
                srv.submit(r)

        t0 = time.perf_counter()
        th = threading.Thread(target=feeder)
        th.start()
        th.join()
        for r in batch:
            r.event.wait(600)
        t1 = time.perf_counter()
        out[f"rate_{f}"] = dict(SolveServer.summarize(batch, t0, t1),
                                offered_per_s=round(f * sat, 2))
    srv.close()
    out["p50_ms"] = out["rate_0.8"]["p50_ms"]
    out["p99_ms"] = out["rate_0.8"]["p99_ms"]
    out["solves_per_s"] = out["saturation"]["solves_per_s"]
    return out


def profile_case(name, dtype):
    """One small case per kernel family for `ncu` captures: inputs larger
    than L2 (129 MB) but a few hundred MB on the device, three launches of
    the kernel after the matrix is built.
      merge    CSR segmented kernel, Zipf(1.8) power-law n=2^21 (~33M nnz)
      coo      COO of the same power-law matrix
      rowtile  CSR row tiles, 3D 7-point Laplacian 128^3 (14.6M nnz)
      warptile CSR warp tiles, the same Laplacian
      ell      ELL of the same Laplacian
      sellp    SELL-P(32) of the same Laplacian
      cg, bicgstab, gmres
               24 Jacobi-preconditioned iterations (GMRES(30): Arnoldi
               steps) on the 128^3 diffusion problem (solver kernels: SpMV
               epilogues, fused updates, multi-dots), the solve graph
               unrolled (GK_SOLVE_UNROLLED=3) so that ncu sees its kernels
      ilu      ILU(0) of the 2D 5-point Laplacian 512^2 and three
               applications (the substitution kernels k_ilu_trsv)
      ilu_banded
               the same on a banded SPD matrix (n = 2^15, half-bandwidth
               48: every row depends on the one before it)"""
    import torch
    import __graft_entry__
    __graft_entry__.build()
    import paper_2510_08230_gb300 as gk
    from paper_2510_08230_gb300 import workloads as W
    dev = torch.device("cuda:0")
    vt = torch.float64 if dtype == "f64" else torch.float32
    if name in ("ilu", "ilu_banded"):
        m = W.laplacian_2d(512) if name == "ilu" else W.banded_spd(1 << 15, 48, 3)
        A = gk.Matrix.from_csr(m, dtype)
        r = torch.from_numpy(W.uniform_vector(m.n, W.SEED_BASE + 3)).to(dev, vt)
        z = torch.empty_like(r)
        for _ in range(3):
            A.precond_apply(r, z, "ilu")
        torch.cuda.synchronize()
        print("profile case", name, dtype, m.n, m.nnz)
        A.close()
        return 0
    if name in ("cg", "bicgstab", "gmres"):
        # the solve graph without its conditional loop node (profilers do not
        # see into such graphs): 3 unrolled passes of 8 iterations
        os.environ["GK_SOLVE_UNROLLED"] = "3"
        m = W.diffusion_3d(128)
        A = gk.Matrix.from_csr(m, dtype)
        b = torch.from_numpy(W.uniform_vector(m.n, W.SEED_BASE + 3)).to(dev, vt)
        x = torch.zeros_like(b)
        info = A.solve(b, x, method=name, precond="jacobi", tol=0.0, max_iters=24)
        torch.cuda.synchronize()
        print("profile case", name, dtype, info["iters"], A.describe()["solve_format"])
        A.close()
        return 0
    if name in ("merge", "coo"):
        os.environ["GK_CSR_KERNEL"] = "2"
        m = W.power_law(1 << 21, seed=W.SEED_BASE + 2)
    else:
        os.environ["GK_CSR_KERNEL"] = "3" if name == "warptile" else "1"
        m = W.laplacian_3d(128)
    A = gk.Matrix.from_csr(m, dtype)
    if name in ("ell", "sellp", "coo"):
        B = A.convert(name, None, 32, 1)
        A.close()
        A = B
    x = torch.from_numpy(np.random.default_rng(1).uniform(-1, 1, m.ncols)).to(dev, vt)
    y = torch.empty(m.n, dtype=vt, device=dev)
    for _ in range(3):
        A.apply(x, y)
    torch.cuda.synchronize()
    print("profile case", name, dtype, KERNEL_NAMES[A.desc["spmv_kernel"]], m.n, m.nnz,
          alg_bytes(m, 8 if dtype == "f64" else 4, "csr" if name in ("merge", "rowtile", "warptile") else name))
    A.close()
    return 0


def run_reference(args):
    """The oracle on the host cores, same metric and unit."""
    rank = int(os.environ.get("RANK", "0"))
    if rank != 0:
        return 0
    from paper_2510_08230_gb300 import workloads as W
    import oracle
    lap = W.laplacian_3d(256)
    rp = np.ascontiguousarray(lap.row_ptr, dtype=np.int32)
    ci = np.ascontiguousarray(lap.col_idx, dtype=np.int32)
    va = np.ascontiguousarray(lap.values, dtype=np.float64)
    x = np.random.default_rng(1).uniform(-1, 1, lap.n)
    y = np.zeros(lap.n)
    nb = alg_bytes(lap, 8, "csr")
    for _ in range(args.warmup):
        oracle.spmv_omp(lap, x, 0, y=y, arrays=(rp, ci, va))
    t0 = time.perf_counter()
    threads = 0
    for _ in range(args.steps):
        _, threads = oracle.spmv_omp(lap, x, 0, y=y, arrays=(rp, ci, va))
    el = time.perf_counter() - t0
    gbs = nb * args.steps / el / 1e9
    sample = (f"each step = 1 FP64 CSR SpMV of the 3D 7-point 256^3 Laplacian by the oracle "
              f"(row-parallel OpenMP, {threads} threads); FP32 / ELL / SELL-P / power-law items "
              f"of the GPU sweep are not run by the oracle")
    line = {"impl": "reference", "metric": METRIC, "value": round(gbs, 3), "unit": "GB/s",
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": round(el * 1000 / args.steps, 3), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "reference_sample": sample},
            "cpu_baseline": {"value": round(gbs, 3), "unit": "GB/s", "cores": threads,
                             "kind": "oracle", "sample": sample},
            "e2e": {"value": round(gbs, 3), "unit": "GB/s", "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# sections that go to stderr alone: the line on stdout has to stay short enough
# for readers that keep the end of a program's output
DETAILS = ("step", "sweep", "cg", "ir_128cubed", "per_iteration_1000", "abi_overhead",
           "preconditioners", "oracle", "batched_2048", "serving")


def headline(line):
    """The result line without its detail sections, with the figures of the
    metric that they hold: CG solves/s and the serving latencies."""
    out = {k: v for k, v in line.items() if k not in DETAILS}
    for section, keys in (("cg", ("solves_per_s",)),
                          ("serving", ("solves_per_s", "p50_ms", "p99_ms"))):
        if line.get(section):
            out[section] = {k: line[section][k] for k in keys if k in line[section]}
    return out


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=10)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="gk", choices=["gk", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-cg", action="store_true")
    ap.add_argument("--no-solvers", action="store_true")
    ap.add_argument("--no-serving", action="store_true")
    ap.add_argument("--profile-case", choices=["merge", "coo", "rowtile", "warptile", "ell",
                                               "sellp", "cg",
                                               "bicgstab", "gmres", "ilu", "ilu_banded"],
                    help="run one small case for an ncu capture and exit")
    ap.add_argument("--profile-dtype", default="f64", choices=["f64", "f32"])
    args = ap.parse_args()
    if args.profile_case:
        return profile_case(args.profile_case, args.profile_dtype)
    if args.impl == "reference":
        return run_reference(args)

    import torch
    import __graft_entry__
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    dev = torch.device(f"cuda:{local}")
    torch.cuda.set_device(dev)
    __graft_entry__.build()
    import paper_2510_08230_gb300 as gk
    from paper_2510_08230_gb300 import workloads as W

    items, lap, pl = build_items(gk, W)
    rng = np.random.default_rng(W.SEED_BASE + 2)
    for it in items:
        vt = torch.float64 if it["dtype"] == "f64" else torch.float32
        it["x"] = torch.from_numpy(rng.uniform(-1, 1, it["ncols"])).to(dev, vt)
        it["y"] = torch.empty(it["n"], dtype=vt, device=dev)
    stream = torch.cuda.current_stream()

    # format choice: fastest format per (matrix, dtype), by a short timing pass
    trial = {it["name"]: time_apply(it, stream, torch) for it in items}
    best = {}
    for it in items:
        key = it["name"].rsplit("/", 2)[0] + "/" + it["dtype"]
        if key not in best or trial[it["name"]] < trial[best[key]["name"]]:
            best[key] = it
    step_items = list(best.values())

    def step(its, events=None):
        for k, it in enumerate(its):
            if events is not None:
                events[k][0].record(stream)
            it["mat"].apply(it["x"], it["y"], stream)
            if events is not None:
                events[k][1].record(stream)

    for _ in range(args.warmup):
        step(step_items)
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    clocks = ClockSampler(local)
    clocks.start()
    time.sleep(0.3)
    evs = [[(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True))
            for _ in step_items] for _ in range(args.steps)]
    t_start = torch.cuda.Event(enable_timing=True)
    t_end = torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    torch.cuda.nvtx.range_push("timed_step")  # lets a profiler capture only the timed launches
    t_start.record(stream)
    for s_ in range(args.steps):
        step(step_items, evs[s_])
    t_end.record(stream)
    torch.cuda.synchronize()
    torch.cuda.nvtx.range_pop()
    if world > 1:
        torch.distributed.barrier()
    clk = clocks.stop()
    total_ms = t_start.elapsed_time(t_end)
    per_item_ms = [statistics.mean(evs[s_][k][0].elapsed_time(evs[s_][k][1])
                                   for s_ in range(args.steps)) for k in range(len(step_items))]
    # the step counts every matrix at its CSR algorithmic bytes, whatever
    # format ran, so a format that moves more (COO's row indices) or less
    # (ELL's missing row pointer) does not change the yardstick
    step_bytes = sum(it["csr_bytes"] for it in step_items)
    total_ms, value = job_throughput(total_ms, step_bytes, args.steps, world, dev)
    peak, peak_kind = _peaks()

    # every format, for the record (not part of the timed step)
    sweep = []
    for it in items:
        ms = time_apply(it, stream, torch, reps=max(3, args.steps))
        gbs = it["bytes"] / (ms / 1000.0) / 1e9
        csr_gbs = it["csr_bytes"] / (ms / 1000.0) / 1e9
        sweep.append({"item": it["name"], "kernel": KERNEL_NAMES[it["kernel"]],
                      "us": round(ms * 1000, 1), "GB_s": round(gbs, 1),
                      "frac_of_measured_hbm": round(gbs / peak, 3),
                      "csr_alg_GB_s": round(csr_gbs, 1),
                      "csr_alg_frac": round(csr_gbs / peak, 3),
                      "frac_of_8TBs_nominal": round(gbs / 8000.0, 3),
                      "in_step": it in step_items})
    # dominant kernel: largest share of the step's device time.  Its
    # algorithmic bytes are the unpadded CSR matrix with x and y once
    # (whatever format ran); the format's own bytes (COO's row index of
    # every entry, padding excluded) are reported beside them.
    k_dom = max(range(len(step_items)), key=lambda k: per_item_ms[k])
    dom = step_items[k_dom]
    dom_s = per_item_ms[k_dom] / 1000.0
    dom_gbs = dom["csr_bytes"] / dom_s / 1e9
    traffic = traffic_for(KERNEL_NAMES[dom["kernel"]], dom["name"])
    roofline = {"bound": "hbm", "achieved": round(dom_gbs, 1), "peak": peak, "unit": "GB/s",
                "frac": round(dom_gbs / peak, 3),
                "traffic": traffic,
                "kernel": KERNEL_NAMES[dom["kernel"]], "item": dom["name"],
                "peak_source": f"{peak_kind} HBM copy bandwidth (MEASURED_PEAKS.json hbm_gbs)"
                if peak_kind == "measured" else "fallback 6.8 TB/s",
                "algorithmic_bytes_per_launch": dom["csr_bytes"],
                "algorithmic_bytes_rule": "CSR: nnz*(sv+4) + 4(n+1) + n*sv (x) + n*sv (y)",
                "format_bytes_per_launch": dom["bytes"],
                "format_frac": round(dom["bytes"] / dom_s / 1e9 / peak, 3),
                "traffic_over_algorithmic": (round(traffic / dom["csr_bytes"], 3)
                                             if traffic else None),
                "mean_launch_us": round(per_item_ms[k_dom] * 1000, 1),
                "share_of_step": round(per_item_ms[k_dom] / sum(per_item_ms), 3)}
    step_detail = [{"item": it["name"], "kernel": KERNEL_NAMES[it["kernel"]],
                    "us": round(ms * 1000, 1),
                    "GB_s": round(it["csr_bytes"] / (ms / 1000.0) / 1e9, 1),
                    "frac_of_measured_hbm": round(it["csr_bytes"] / (ms / 1000.0) / 1e9 / peak, 3)}
                   for it, ms in zip(step_items, per_item_ms)]

    # e2e: the same step through the C ABI with pinned HOST buffers (H2D of
    # x, kernel, D2H of y inside the timed region, every step).  gk_apply
    # with host vectors blocks until y is back; calls on different handles
    # may run concurrently (gk.h), so each matrix gets its own host thread
    # and CUDA stream and the host link carries both directions at once
    # while kernels run.
    import concurrent.futures as cf
    hx = [torch.from_numpy(it["x"].cpu().numpy()).pin_memory() for it in step_items]
    hy = [torch.empty(it["n"], dtype=it["y"].dtype).pin_memory() for it in step_items]
    e2e_streams = [torch.cuda.Stream() for _ in step_items]
    pool = cf.ThreadPoolExecutor(max_workers=len(step_items))

    def one(k):
        torch.cuda.set_device(dev)
        step_items[k]["mat"].apply(hx[k], hy[k], e2e_streams[k])

    def e2e_step():
        for f in [pool.submit(one, k) for k in range(len(step_items))]:
            f.result()

    e2e_step()
    torch.cuda.synchronize()
    if world > 1:
        torch.distributed.barrier()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        e2e_step()
    torch.cuda.synchronize()
    e2e_s = time.perf_counter() - t0
    pool.shutdown()
    _, e2e_gbs = job_throughput(e2e_s * 1000.0, step_bytes, args.steps, world, dev)
    h2d = sum(a.numel() * a.element_size() for a in hx)
    d2h = sum(b.numel() * b.element_size() for b in hy)
    e2e = {"value": round(e2e_gbs, 1), "unit": "GB/s",
           "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
           "how": "gk_apply with pinned host x and y (library-staged copies), one host thread "
                  "and CUDA stream per matrix, host wall clock"}
    launches = sum(it["launches"] for it in step_items) * args.steps
    for it in items:
        it["mat"].close()
    del items, step_items
    torch.cuda.empty_cache()

    cg = ir = batched = serving = per_iter = abi = pre = orc = None
    keep = {}
    if rank == 0 and not args.no_cg:
        cg = cg_solves_per_s(gk, W, torch, dev, keep=keep)
    if rank == 0 and not args.no_solvers:
        ir = ir_compare(gk, W, torch, dev, keep=keep)
        per_iter = per_iteration_protocol(gk, W, torch, dev)
        abi = abi_overhead(gk, W, torch, dev)
        pre = precond_compare(gk, W, torch, dev, keep=keep)
        batched = batched_compare(gk, W, torch, dev, keep=keep)
    if rank == 0 and not args.no_serving:
        serving = serving_bench(gk, W, torch, dev)
    cpu = None
    if not args.no_cpu_baseline and rank == 0 and world == 1:
        cpu = cpu_baseline(lap)
        orc = oracle_legs(W, lap, keep)
    del keep
    line = {"metric": METRIC, "value": round(value, 1), "unit": "GB/s", "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": round(total_ms / args.steps, 3), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64+f32", "data": "synthetic",
            "config": {"workload": WORKLOAD, "l2": "inputs larger than L2 (no flush)",
                       "parallelism": f"replicas x{world}" if world > 1 else "1 GPU"},
            "step": step_detail, "sweep": sweep, "roofline": roofline, "cpu_baseline": cpu,
            "e2e": e2e, "cg": cg, "ir_128cubed": ir, "per_iteration_1000": per_iter,
            "abi_overhead": abi, "preconditioners": pre, "oracle": orc,
            "batched_2048": batched,
            "serving": serving, "clocks": clk,
            "gpu_launches": launches}
    if rank == 0:
        print(json.dumps(line), file=sys.stderr, flush=True)  # every section in full
        print(json.dumps(headline(line)), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()
    return 0


if __name__ == "__main__":
    sys.exit(main())
