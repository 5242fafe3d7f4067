#!/usr/bin/env python
"""Benchmark: Gauss-Newton Hessian actions per second at relative residual 1e-8.

One step = one block of k+p Gauss-Newton Hessian actions (the block the
double-pass eigensolver applies, Algorithm 2) at the MAP point of a seeded
synthetic problem: per column one incremental forward and one incremental
adjoint solve (FP32 multigrid PCG inside FP64 iterative refinement, every
column to relative residual 1e-8), plus the C X, B^T B and C^T kernels.
Inputs are resident on the device; L2 is flushed (a 512 MB write) before every
timed step and each step is timed with CUDA events on the library's stream.

Also reported: e2e (same metric through the C ABI with the block copied from
pinned host memory and the result read back inside the timed region), the
time to MAP (Newton-CG, Algorithm 1) plus the rank-k eigenpairs (Algorithm 2),
the roofline of the dominant kernel measured live with CUDA events, clocks
sampled during the timed region, and the FP64 CPU oracle on a bounded sample.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]
                    [--workload cube3d|medium2d|small2d|batch64] [--precision fp32_ir|fp64]

The default workload is cube3d (64^3 Kuhn tetrahedra, 274,625 nodes, 120 columns): the
largest single-GPU configuration, whose blocks do not fit in L2.
"""
from __future__ import annotations

import os

os.environ.setdefault("OMP_NUM_THREADS", "1")
os.environ.setdefault("OPENBLAS_NUM_THREADS", "1")
os.environ.setdefault("MKL_NUM_THREADS", "1")
# 32 hardware work queues for the batch's per-problem streams (the CUDA default is 8); read
# when CUDA starts, so it is set before anything touches the GPU
os.environ.setdefault("CUDA_DEVICE_MAX_CONNECTIONS", "32")

import argparse
import hashlib
import json
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)
import workloads as W  # noqa: E402

METRIC = "Hessian actions/s at rel-res 1e-8"
FALLBACK_HBM_GBS = 6800.0


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="cube3d", choices=sorted(W.WORKLOADS) + ["batch64"])
    ap.add_argument("--precision", default="fp32_ir", choices=["fp32_ir", "fp64"])
    ap.add_argument("--no-map", action="store_true", help="linearise at the true parameter instead of the MAP")
    ap.add_argument("--no-cpu", action="store_true", help="skip the CPU-oracle baseline leg")
    ap.add_argument("--no-warmstart", action="store_true", help="skip the learned warm-start leg (2D)")
    ap.add_argument("--no-autotune", action="store_true",
                    help="use the library's default solver settings instead of the autotuned ones")
    ap.add_argument("--tuning", default="",
                    help="fixed solver settings instead of the autotuned ones, as key=value pairs separated by "
                         "commas (hp_tuning member names, e.g. tma_tiles=1,col_chunk=32); unnamed members keep "
                         "the library defaults")
    ap.add_argument("--no-plain", action="store_true",
                    help="skip the plain one-vector FP64 GPU path (the speedup denominator)")
    ap.add_argument("--ws-draws", type=int, default=12, help="prior draws whose solves train the warm start")
    ap.add_argument("--ws-epochs", type=int, default=8, help="training epochs of the warm start")
    return ap.parse_args()


def parse_tuning(text):
    """{'name': number} from "name=value,name=value" (integers where the value is one)."""
    out = {}
    for item in filter(None, (t.strip() for t in text.split(","))):
        key, _, val = item.partition("=")
        if not key or not val:
            raise SystemExit(f"--tuning: expected name=value, got {item!r}")
        try:
            out[key.strip()] = int(val)
        except ValueError:
            out[key.strip()] = float(val)
    return out


def workload_desc(w, precision):
    prec = {"fp32_ir": "FP32 MG-PCG in FP64 refinement", "fp64": "FP64 MG-PCG",
            "oracle_direct": "FP64 CPU oracle with sparse direct solves (exact to rounding)",
            "oracle_cg": "FP64 CPU oracle with Jacobi-preconditioned CG solves to relative residual 1e-13"}[precision]
    return (f"{w.name}: {w.dim}D {'x'.join([str(w.N)] * w.dim)} P1 "
            f"({'right triangles' if w.dim == 2 else 'Kuhn tetrahedra'}), n={w.nnodes}, q={w.nobs}, "
            f"block of k+p={w.k + w.p} Gauss-Newton Hessian actions at the MAP, {prec}, rel-res 1e-8")


# ---------------------------------------------------------------------------
# CPU oracle leg (the only place besides --impl reference that runs oracle/)
# ---------------------------------------------------------------------------
def oracle_rate(w, ncols_sample, seconds_hint=20.0):
    """Oracle Hessian actions/s for a (k+p)-column block, from a bounded sample: the
    linearisation point's set-up (2D: one sparse direct factorisation of K(m); 3D: none,
    every solve is a Jacobi-preconditioned CG) + ncols_sample columns, extrapolated to the
    full block."""
    from oracle.inverse import make_problem
    dr = W.draws(w)
    prob, m_true, _ = make_problem(w, dr)
    m = m_true
    s_full = w.k + w.p
    X = W.omega(w)
    t0 = time.perf_counter()
    u = prob.forward(m)                       # 2D: factorises K(m); 3D: one CG solve
    t_fac = time.perf_counter() - t0 if prob.solver == "direct" else 0.0
    cols = 0
    t1 = time.perf_counter()
    while cols < ncols_sample:
        prob.hessian_misfit(m, u, X[:, cols:cols + 1])
        cols += 1
        if time.perf_counter() - t1 > seconds_hint:
            break
    t_cols = time.perf_counter() - t1
    per_col = t_cols / cols
    block_time = t_fac + s_full * per_col
    return s_full / block_time, cols, t_fac, per_col


ORACLE_SOLVES = {
    "direct": "sparse direct solves (SuperLU), exact to rounding",
    "cg": "Jacobi-preconditioned CG solves to relative residual 1e-13 (a sparse direct factorisation does not "
          "finish in minutes on 3D meshes of this size)",
}


def host_cores():
    return os.cpu_count() or 1


def cpu_baseline_block(w):
    ncols = {"small2d": 30, "medium2d": 8, "cube3d": 1}[w.name]
    rate, cols, t_fac, per_col = oracle_rate(w, ncols)
    kind = "cg" if w.dim == 3 else "direct"
    setup = (f"one K(m) factorisation ({t_fac:.2f} s) + " if kind == "direct" else "")
    return {"value": rate, "unit": "actions/s", "cores": 1, "host_cores": host_cores(), "kind": "oracle",
            "sample": (f"FP64 numpy/scipy oracle ({ORACLE_SOLVES[kind]}), {setup}{cols} of {w.k + w.p} columns "
                       f"({per_col:.2f} s each), extrapolated to the {w.k + w.p}-column block; 1 thread of "
                       f"{host_cores()} host cores")}


def oracle_batch_rate(ws, every=8, ncols=1):
    """Oracle Hessian actions/s for the batch of independent problems, from a bounded
    sample: every `every`-th problem (one K(m) factorisation + `ncols` columns, extrapolated
    to its k+p-column block); the sampled block times, scaled by len(ws) / samples, stand
    for the whole batch run one problem after another."""
    from oracle.inverse import make_problem
    t_blocks, sampled = 0.0, 0
    for w in ws[::every]:
        prob, m, _ = make_problem(w, W.draws(w))
        X = W.omega(w)
        t0 = time.perf_counter()
        u = prob.forward(m)
        t_fac = time.perf_counter() - t0
        t1 = time.perf_counter()
        prob.hessian_misfit(m, u, X[:, :ncols])
        per_col = (time.perf_counter() - t1) / ncols
        t_blocks += t_fac + (w.k + w.p) * per_col
        sampled += 1
    units = sum(w.k + w.p for w in ws)
    return units / (t_blocks * len(ws) / sampled), sampled


def run_reference(args, rank, world):
    if rank != 0:
        return
    if args.workload == "batch64":
        ws = W.batch_workloads(seed=W.SEED_BASE + 3)
        t0 = time.perf_counter()
        val, sampled = oracle_batch_rate(ws)
        dt = time.perf_counter() - t0
        sample = (f"{sampled} of {len(ws)} problems (every 8th): set-up, one K(m) factorisation and one "
                  f"Hessian-action column each, extrapolated to the problems' 40-column blocks and to the "
                  f"whole batch run one problem after another, 1 thread ({dt:.0f} s)")
        print(json.dumps({
            "impl": "reference", "metric": METRIC, "value": val, "unit": "actions/s", "n_gpus": args.gpus,
            "steps": 1, "warmup": 0, "ms_per_step": 1e3 * sum(w.k + w.p for w in ws) / val,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": f"batch64: {len(ws)} independent 2D problems, one block of k+p=40 GN Hessian "
                                   f"actions per problem, FP64 CPU oracle with sparse direct solves",
                       "l2": "n/a (CPU)"},
            "cpu_baseline": {"value": val, "unit": "actions/s", "cores": 1, "host_cores": host_cores(),
                             "kind": "oracle", "sample": sample},
            "e2e": {"value": val, "unit": "actions/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
            "gpu_launches": 0}), flush=True)
        return
    w = W.WORKLOADS[args.workload]
    from oracle.inverse import make_problem
    dr = W.draws(w)
    prob, m_true, _ = make_problem(w, dr)
    m = m_true
    X = W.omega(w)
    s_ref = {"small2d": 10, "medium2d": 2, "cube3d": 1}[w.name]
    u = prob.forward(m)
    # the oracle keeps nothing between steps, so one warm-up step stands for any number
    warm = min(args.warmup, 1) if prob.solver == "cg" else args.warmup
    for i in range(warm):
        prob.hessian_misfit(m, u, X[:, :s_ref])
    t0 = time.perf_counter()
    for i in range(args.steps):
        prob.hessian_misfit(m, u, X[:, (i * s_ref) % (w.k + w.p):(i * s_ref) % (w.k + w.p) + s_ref])
    dt = time.perf_counter() - t0
    val = args.steps * s_ref / dt
    line = {
        "impl": "reference", "metric": METRIC, "value": val, "unit": "actions/s", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": warm, "ms_per_step": 1e3 * dt / args.steps,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": workload_desc(w, "oracle_" + prob.solver) + f"; reference arm: {s_ref} column(s) "
                                                                            f"per step",
                   "l2": "n/a (CPU)"},
        "cpu_baseline": {"value": val, "unit": "actions/s", "cores": 1, "host_cores": host_cores(), "kind": "oracle",
                         "sample": (f"{s_ref} Hessian-action column(s) per step, " +
                                    ("K(m) factorised once before the warm-up" if prob.solver == "direct" else
                                     "every solve a Jacobi-preconditioned CG to 1e-13") +
                                    f"; 1 thread of {host_cores()} host cores")},
        "e2e": {"value": val, "unit": "actions/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "gpu_launches": 0,
    }
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------------------
# GPU leg
# ---------------------------------------------------------------------------
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.path = tempfile.mktemp(prefix="hp_clocks_", suffix=".csv")
        self.proc = None
        try:
            self.f = open(self.path, "w")
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(gpu_index), f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "50"],
                                         stdout=self.f, stderr=subprocess.DEVNULL)
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
            for nm, v in zip(names, parts[5:9]):
                if v.lower() == "active":
                    reasons.add(nm)
        os.unlink(self.path)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def build_record():
    """Which machine and compiler built the loaded libhp.so (build.py's stamp) and when: the
    library is rebuilt whenever the stamp differs from the machine it runs on."""
    pkg = os.path.join(ROOT, "paper_1909_03948_gb300")
    out = {"machine": os.uname().machine}
    try:
        stamp = open(os.path.join(pkg, "_build", "STAMP")).read().split("\n")
        out["built_on"], out["nvcc"] = stamp[0], stamp[1] if len(stamp) > 1 else None
        out["lib_mtime"] = time.strftime("%Y-%m-%dT%H:%M:%S", time.gmtime(os.path.getmtime(os.path.join(pkg, "libhp.so"))))
    except OSError as ex:
        out["error"] = str(ex)
    return out


def measured_peak():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        try:
            d = json.load(open(p))
            for key in ("hbm_gbs", "hbm_GBs", "hbm"):
                if key in d:
                    return float(d[key]), "measured (MEASURED_PEAKS.json hbm_gbs)"
        except Exception:
            pass
    return FALLBACK_HBM_GBS, "fallback (6.8 TB/s recipe figure; MEASURED_PEAKS.json absent)"


def family_bytes(fam, n, s, dim, fp32):
    """Algorithmic DRAM bytes of one launch of a level-0 kernel family on n nodes x s columns."""
    w = 4 if fp32 else 8
    nf = dim  # forward couplings of the stiffness stencil
    if fam == "matvec":       # read p, write q, coefficients (diag + nf)
        return n * (2 * s * w + (nf + 1) * w)
    if fam == "smooth":       # read x, b, write y, coefficients (diag, invdiag, nf)
        return n * (3 * s * w + (nf + 2) * w)
    if fam == "presmooth":    # two fused sweeps from zero: read r, write e, coefficients
        return n * (2 * s * w + (nf + 2) * w)
    if fam == "resid_mg":     # read x, b, write r, coefficients
        return n * (3 * s * w + (nf + 1) * w)
    if fam == "resid64":      # FP64 refinement residual
        return n * (3 * s * 8 + (nf + 1) * 8)
    if fam == "cg_update":    # read p, q, x, r; write x, r
        return n * 6 * s * w
    if fam == "leg_down":     # read r, write e and the coarse right-hand side, coefficients
        return n * (2 * s * w + (nf + 2) * w) + (n * s * w) // 2 ** dim
    if fam == "leg_up":       # read e, r and the coarse correction, write e, coefficients
        return n * (3 * s * w + (nf + 2) * w) + (n * s * w) // 2 ** dim
    if fam == "columns":      # read r, write x (the rest stays on chip)
        return n * 2 * s * w
    if fam == "cheb_step":    # read x, the iterate before it and b, write y, coefficients of all edges
        return n * (4 * s * w + (2 ** dim + 1) * w)
    return None


def stencil_kernel_sha256(kind="row"):
    """sha256 of a level-0 stencil kernel's source (the code an ncu traffic record belongs
    to), with csrc/common.cuh.  kind "row": the Pack / reduction / k_st block of
    csrc/solver.cu up to the tiled kernels; kind "tiled": the TMA-tiled kernels k_st_tile and
    k_st_tile3 with the tile shapes of csrc/internal.h."""
    csrc = os.path.join(ROOT, "paper_1909_03948_gb300", "csrc")
    src = open(os.path.join(csrc, "solver.cu")).read()
    if kind == "row":
        a = src.index("template <typename T, int VW> struct Pack {")
        b = src.index("// TMA-tiled stencil kernels")
        h = hashlib.sha256(src[a:b].encode())
    else:
        a = src.index("// TMA-tiled stencil kernels")
        b = src.index("// grid transfer, coarse solve")
        h = hashlib.sha256(src[a:b].encode())
        hdr = open(os.path.join(csrc, "internal.h")).read()
        h.update(hdr[hdr.index("// Grids whose stiffness stencils run as TMA-tiled kernels"):
                     hdr.index("// Symmetric stencil stored")].encode())
    h.update(open(os.path.join(csrc, "common.cuh"), "rb").read())
    return h.hexdigest()


def level0_kernel_kind(dim, N, tune, fp32):
    """"tiled" when the level-0 stiffness sweeps run as TMA-tiled kernels, else "row": the
    tiled kernels are FP32, enabled by the tma_tiles setting, and take grids whose N is a
    multiple of the tile (32 x 16 in 2D; 32 x 8 xy tiles and 16-plane z segments in 3D)."""
    if not (fp32 and tune and tune.get("tma_tiles")) or N < 32:
        return "row"
    ok = N % 32 == 0 and N % 16 == 0 if dim == 2 else N % 32 == 0 and N % 8 == 0 and N % 16 == 0
    return "tiled" if ok else "row"


def traffic_record(fam, workload, kind="row", path=None):
    """ncu DRAM bytes per launch recorded in profiles/traffic.json (or ``path``) for a
    level-0 kernel family, valid only for the kernel form that ran (row or tiled) while
    that kernel's source is unchanged (stencil_kernel_sha256)."""
    p = path or os.path.join(ROOT, "profiles", "traffic.json")
    if not os.path.exists(p):
        return None
    try:
        d = json.load(open(p))
        rec = d.get(workload, {}).get(fam)
        if rec and rec.get("kind", "row") == kind and rec.get("src_sha256") == stencil_kernel_sha256(kind):
            return rec.get("dram_bytes_per_launch")
    except Exception:
        return None
    return None


def weak_scaling_value(t_local, units_per_rank, world, device="cpu"):
    """Whole-job throughput for replicas on `world` ranks: every rank processes
    units_per_rank units; the job takes the slowest rank's time (max over ranks)."""
    t_max = float(t_local)
    if world > 1:
        import torch
        import torch.distributed as dist
        t = torch.tensor([t_local], dtype=torch.float64, device=device)
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
        t_max = float(t)
    return world * units_per_rank / t_max, t_max


def run_ours(args, rank, world):
    import torch
    from paper_1909_03948_gb300 import Problem, algorithmic_bytes, kernel_launches

    torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", "0")))
    dev = torch.device("cuda", torch.cuda.current_device())
    w = W.WORKLOADS[args.workload]
    wr = W.Workload(**{**w.__dict__, "seed": w.seed + 1000 * rank})     # weak scaling: own replica per rank
    dr = W.draws(wr)
    s = w.k + w.p
    # ---- problem set-up (untimed): synthetic truth and data on the GPU path ----
    P = Problem(w.dim, w.N, w.gamma, w.delta, 1.0, dr.obs_xyz, precision=args.precision, rtol=1e-8)
    eta = torch.tensor(dr.eta_true.reshape(1, -1), device=dev)
    m_true, _, _ = P.laplace_sample(None, None, None, eta, want_prior=True, want_post=False)
    m_true = m_true[0].contiguous()
    u_true, _ = P.forward(m_true)
    sigma = w.noise_level * float(u_true.abs().max())
    d = P.observe(u_true).cpu().numpy() + sigma * dr.xi_noise
    P.set_data(d, sigma)
    Omega = torch.tensor(np.ascontiguousarray(W.omega(wr).T), device=dev)
    # ---- time to MAP + rank-k eigenpairs (once) ----
    extra = {}
    if not args.no_map:
        # Newton-CG with its CG preconditioned by R^-1 only (Section 4.1), then with the
        # low-rank correction from block eigensolves (k + p actions per refresh, every 2
        # Newton iterations); the second is the timed path of this build
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        m_r, nst_r = P.newton_cg_map(rel_tol=1e-6)
        P.lowrank_eig(m_r, w.k, w.p, Omega)
        torch.cuda.synchronize()
        t_rinv = time.perf_counter() - t0
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        m_map, nst = P.newton_cg_map(rel_tol=1e-6, lowrank_k=w.k, lowrank_p=w.p, lowrank_refresh=2)
        lam, V, est = P.lowrank_eig(m_map, w.k, w.p, Omega)
        torch.cuda.synchronize()
        t_me = time.perf_counter() - t0
        extra = {"time_to_map_eig_s": t_me, "newton_iterations": nst["iterations"],
                 "newton_cg_iterations": nst["cg_iterations"], "newton_eig_refreshes": nst["eig_solves"],
                 "newton_converged": bool(nst["converged"]),
                 "newton_preconditioner": f"R^-1 - V D V^T, {w.k} eigenpairs refreshed every 2 Newton iterations",
                 "time_to_map_eig_s_rinv_only": t_rinv, "newton_cg_iterations_rinv_only": nst_r["cg_iterations"],
                 "lambda_1": float(lam[0]), "lambda_k": float(lam[-1])}
        if w.nsamples:
            # Laplace-approximation samples at the MAP (Section 4.3), normals drawn on the device
            P.laplace_sample(m_map, lam, V, None, seed=w.seed, nsamples=min(w.nsamples, 64))
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            _, post, sst = P.laplace_sample(m_map, lam, V, None, seed=w.seed + 1, nsamples=w.nsamples,
                                            want_prior=True)
            torch.cuda.synchronize()
            t_s = time.perf_counter() - t0
            extra["laplace_samples"] = {"n": w.nsamples, "seconds": t_s, "samples_per_s": w.nsamples / t_s,
                                        "prior_solve_iterations": sst["iterations"]}
            del post
        m_lin = m_map
    else:
        m_lin = m_true
    P.set_point(m_lin)
    from paper_1909_03948_gb300 import tuning
    if args.tuning:
        fixed = parse_tuning(args.tuning)
        P.set_tuning(**fixed)
        tune, tune_ms, tune_src = P.get_tuning(), None, f"library defaults with {args.tuning}"
    elif args.no_autotune:
        P.set_tuning()
        tune, tune_ms, tune_src = P.get_tuning(), None, "library defaults"
    else:
        # tuned on the timed block itself: a candidate's PCG iteration count depends on the
        # right-hand sides, so a random block can favour another smoother
        tune, tune_ms, tune_src = tuning.tuned(P, s, args.precision, X=Omega)
    Y = torch.empty_like(Omega)
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)

    def step():
        return P.hessian_apply(Omega, out=Y)[1]

    for _ in range(max(args.warmup, 3)):
        st = step()
    # ---- timed region (device-resident inputs) ----
    if world > 1:
        torch.distributed.barrier()
    torch.cuda.synchronize()
    clocks = ClockSampler(torch.cuda.current_device())
    l0 = kernel_launches()
    times, iters, outers = [], [], []
    for _ in range(args.steps):
        flush.fill_(1.0)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        st = step()
        e1.record()
        e1.synchronize()
        times.append(e0.elapsed_time(e1) / 1e3)
        iters.append(st["iterations"])
        outers.append(st["outer"])
    torch.cuda.synchronize()
    launches = kernel_launches() - l0
    clk = clocks.stop()
    t_total = sum(times)
    # ---- same K steps again with CUDA events around the level-0 kernels (roofline) ----
    # (direct launches: the library also counts every launch's algorithmic bytes here)
    P.profile_enable(True)
    t_prof = 0.0
    b0, lp0 = algorithmic_bytes(), kernel_launches()
    for _ in range(args.steps):
        flush.fill_(1.0)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        step()
        e1.record()
        e1.synchronize()
        t_prof += e0.elapsed_time(e1) / 1e3
    prof = P.profile_read()
    P.profile_enable(False)
    b1, lp1 = algorithmic_bytes(), kernel_launches()
    step_bytes = {k: (b1[k] - b0[k]) / args.steps for k in b0}
    launches_direct = lp1 - lp0
    value, t_total = weak_scaling_value(t_total, args.steps * s, world, dev)
    # ---- e2e through the C ABI with host buffers ----
    Xh = torch.empty((s, P.n), dtype=torch.float64).pin_memory()
    Xh.copy_(Omega.cpu())
    Yh = torch.empty_like(Xh).pin_memory()
    Xd = torch.empty_like(Omega)
    e2e_times = []
    for _ in range(args.steps):
        flush.fill_(1.0)
        torch.cuda.synchronize()
        ta = time.perf_counter()
        Xd.copy_(Xh, non_blocking=True)
        P.hessian_apply(Xd, out=Y)
        Yh.copy_(Y, non_blocking=False)
        e2e_times.append(time.perf_counter() - ta)
    e2e_val = weak_scaling_value(sum(e2e_times), args.steps * s, world, dev)[0] if e2e_times else None
    # ---- roofline of the dominant level-0 kernel family ----
    fams = {k: v for k, v in prof.items() if k != "vcycle" and v[0] > 0}
    dom = max(fams, key=lambda k: fams[k][1]) if fams else None
    roof = None
    if dom:
        cnt, ms = fams[dom]
        fp32 = args.precision == "fp32_ir" and dom != "resid64"
        bpl = family_bytes(dom, P.n, s, w.dim, fp32)
        kind = ("vector" if dom == "cg_update" else "leg" if dom.startswith("leg") else
                "column" if dom == "columns" else level0_kernel_kind(w.dim, w.N, tune, fp32))
        in_step_s = ms / cnt / 1e3
        peak, src = measured_peak()
        warm_us = cold_us = graph_us = None
        if fp32 and dom in P.REPLAY_FAMILIES:
            # the same launch replayed on the live workspace: back to back (L2-warm), and
            # each launch after a 512 MB read (HBM-cold) minus the reads timed alone; and
            # 200 launches captured in one CUDA graph, as the solver's PCG loop runs them
            P.replay_kernel(dom, 5, flush)
            warm_us, cold_us = P.replay_kernel(dom, 50, flush)
            graph_us = P.replay_kernel_graph(dom, 200)
        # the launch duration is the kernel's as the timed step runs it: a node of a CUDA graph
        # on the live workspace; the per-launch events of the direct-launch pass are kept beside
        # it (stream launches come in steps of about 2 us and carry the event pair's overhead)
        dur_s = graph_us * 1e-6 if graph_us else in_step_s
        ach = bpl / dur_s / 1e9
        roof = {"bound": "hbm", "achieved": ach, "peak": peak, "unit": "GB/s", "frac": ach / peak,
                "traffic": traffic_record(dom, w.name, kind), "kernel": dom, "kernel_form": kind, "launches": cnt,
                "avg_launch_us": dur_s * 1e6, "algorithmic_bytes_per_launch": bpl, "peak_source": src,
                "measured_in": ("the step's own level-0 launch, 200 launches captured in one CUDA graph on the live "
                                "workspace after the timed region, CUDA events around the graph launch "
                                "(replay_us.in_graph)" if graph_us else
                                "a second pass of the same K steps with direct launches, CUDA events around each "
                                "launch"),
                "in_step_direct_launch_us": in_step_s * 1e6,
                "in_step_how": ("a second pass of the same K steps with direct launches, CUDA events around each "
                                "launch (the event pair's own overhead included), each PCG iteration headed by a "
                                "bounded spin so kernels run back to back"),
                "replay_us": {"l2_warm": warm_us, "hbm_cold": cold_us, "in_graph": graph_us,
                              "how": ("the step's own level-0 launch repeated 50 times on the live workspace: back "
                                      "to back, and each after a 512 MB L2-evicting read minus the reads alone; "
                                      "in_graph: 200 launches captured in one CUDA graph (stream launches back "
                                      "to back come in steps of about 2 us, graph nodes do not)")},
                "share_of_step": ms / 1e3 / t_prof,
                "families": {k: {"launches": v[0], "ms": v[1]} for k, v in prof.items()}}
        # fractions of the other two durations, beside the in-graph one
        roof["frac_in_step_direct_launch"] = bpl / in_step_s / 1e9 / peak
        if cold_us:
            roof["frac_hbm_cold_replay"] = bpl / (cold_us * 1e-6) / 1e9 / peak
        # working set of the inner solves: 5 FP32 blocks plus about 1.4 blocks for the coarser
        # levels; while it fits in the 129 MB L2, kernels between flushes run from L2
        ws = 6.4 * P.n * s * 4
        roof["working_set_mb"] = ws / 1e6
        roof["residency"] = ("L2-resident (the in-graph figure is an L2 replay, not an HBM one)"
                             if ws < 120e6 else "spills L2 (HBM-bound)")
        # step level: every launch's algorithmic bytes in one step over the timed step's duration
        tot = sum(step_bytes.values())
        ms_step = 1e3 * t_total / args.steps
        roof["step"] = {
            "achieved": tot / (ms_step * 1e-3) / 1e9, "peak": peak, "unit": "GB/s",
            "frac": tot / (ms_step * 1e-3) / 1e9 / peak, "bytes_per_step": tot, "ms_per_step": ms_step,
            "families": {k: {"bytes_per_step": v, "share_of_bytes": v / tot if tot else None}
                         for k, v in step_bytes.items()},
            "how": ("algorithmic bytes of every launch in a step (each array a kernel must read or write, once per "
                    "launch; counted by the library on the direct-launch pass, which runs the same kernels and "
                    "iterations as the graph-driven timed steps) over the timed steps' mean duration"),
            "launches_per_step_direct": launches_direct / args.steps,
            "launches_per_step_timed": launches / args.steps}
    if rank != 0:
        return
    if not args.no_plain:
        try:
            extra["plain_fp64_one_vector"] = plain_fp64_leg(w, wr, dev, Omega, m_lin, extra.get("time_to_map_eig_s"),
                                                             value, args)
        except Exception as ex:  # pragma: no cover
            extra["plain_fp64_one_vector"] = {"failed": str(ex)}
    if w.dim == 2 and not args.no_warmstart:
        try:
            extra["warm_start"] = warmstart_leg(P, Omega, m_lin, args, dev)
        except Exception as ex:  # pragma: no cover
            extra["warm_start"] = {"failed": str(ex)}
    cpu = None
    if not args.no_cpu and world == 1:
        try:
            cpu = cpu_baseline_block(w)
        except Exception as ex:  # pragma: no cover
            cpu = {"value": None, "unit": "actions/s", "cores": 1, "kind": "oracle", "sample": f"failed: {ex}"}
    line = {
        "metric": METRIC, "value": value, "unit": "actions/s", "n_gpus": world, "steps": args.steps,
        "warmup": max(args.warmup, 3), "ms_per_step": 1e3 * t_total / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32-in-f64-IR" if args.precision == "fp32_ir" else "f64",
        "data": "synthetic (seeded prior draw, pointwise observations with 1% noise)",
        "config": {"workload": workload_desc(w, args.precision), "block_columns": s,
                   "l2": "flushed (512 MB write) before every timed step", "replicas": world,
                   "tuning": {**tune, "source": tune_src}},
        "e2e": {"value": e2e_val, "unit": "actions/s", "h2d_bytes_per_step": s * P.n * 8,
                "d2h_bytes_per_step": s * P.n * 8},
        "gpu_launches": launches,
        "clocks": clk,
        "roofline": roof,
        "cpu_baseline": cpu,
        "pcg": {"inner_iterations_per_step": statistics.median(iters), "refinement_steps": statistics.median(outers)},
        "build": build_record(),
        **extra,
    }
    print(json.dumps(line), flush=True)


def synthetic_problem(w, dev, precision="fp32_ir"):
    """GPU-side synthetic instance: truth = prior draw from the workload's normals,
    data = B u(truth) + sigma xi with sigma = 1 % of max|u|."""
    import torch
    from paper_1909_03948_gb300 import Problem
    dr = W.draws(w)
    P = Problem(w.dim, w.N, w.gamma, w.delta, 1.0, dr.obs_xyz, precision=precision, rtol=1e-8)
    eta = torch.tensor(dr.eta_true.reshape(1, -1), device=dev)
    m_true = P.laplace_sample(None, None, None, eta, want_prior=True, want_post=False)[0][0].contiguous()
    u_true, _ = P.forward(m_true)
    sigma = w.noise_level * float(u_true.abs().max())
    P.set_data(P.observe(u_true).cpu().numpy() + sigma * dr.xi_noise, sigma)
    return P


def plain_fp64_leg(w, wr, dev, Omega, m_lin, t_me, value, args):
    """The plain one-vector FP64 GPU path on the same GPU: the same kernels with
    FP64 multigrid-preconditioned CG throughout (no FP32 inner solver, no refinement),
    one right-hand side per solve, untuned.  Measures Gauss-Newton actions/s on a bounded
    number of single columns, and time to MAP + rank-k eigenpairs."""
    import torch
    from paper_1909_03948_gb300 import Problem
    dr = W.draws(wr)
    P = Problem(w.dim, w.N, w.gamma, w.delta, 1.0, dr.obs_xyz, precision="fp64", rtol=1e-8)
    eta = torch.tensor(dr.eta_true.reshape(1, -1), device=dev)
    m_true = P.laplace_sample(None, None, None, eta, want_prior=True, want_post=False)[0][0].contiguous()
    u_true, _ = P.forward(m_true)
    sigma = w.noise_level * float(u_true.abs().max())
    P.set_data(P.observe(u_true).cpu().numpy() + sigma * dr.xi_noise, sigma)
    P.set_tuning(nu=2, omega=0.7, smoother=0, col_chunk=1)
    out = {"precision": "fp64 MG-PCG, one column per solve (col_chunk 1), damped Jacobi nu 2, untuned"}
    P.set_point(m_lin)
    ncol = min(8, Omega.shape[0])
    P.hessian_apply(Omega[0].contiguous())
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for j in range(ncol):
        P.hessian_apply(Omega[j].contiguous())
    torch.cuda.synchronize()
    t = (time.perf_counter() - t0) / ncol
    out["actions_per_s"] = 1.0 / t
    out["speedup_actions_per_s"] = value / out["actions_per_s"]
    if t_me is not None and not args.no_map:
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        m_map, nst = P.newton_cg_map(rel_tol=1e-6)
        # one column at a time: the double pass needs k + p actions per pass
        lam, V, _ = P.lowrank_eig(m_map, w.k, w.p, Omega)
        torch.cuda.synchronize()
        out["time_to_map_eig_s"] = time.perf_counter() - t0
        out["speedup_time_to_map_eig"] = out["time_to_map_eig_s"] / t_me
        out["newton_iterations"] = nst["iterations"]
    P.close()
    return out


def warmstart_leg(P, Omega, m_lin, args, dev):
    """Learned warm start against the zero start on the bench's own block of Hessian
    actions: train the network on the solves of fresh prior draws (recorded by the
    library), then time the block and count PCG iterations with and without it."""
    import torch
    from paper_1909_03948_gb300.warmstart import generate, prior_draws, train
    t0 = time.perf_counter()
    ms = prior_draws(P, args.ws_draws, seed=4242)
    X, A = generate(P, ms, ncols=16, seed=4343)
    t_gen = time.perf_counter() - t0
    t0 = time.perf_counter()
    net, losses = train(X, A, epochs=args.ws_epochs, batch=16, lr=1e-3, seed=7)
    torch.cuda.synchronize()
    t_train = time.perf_counter() - t0
    nsamp = X.shape[0]
    del X, A
    s = Omega.shape[0]
    Y = torch.empty_like(Omega)
    out = {}
    for on in (False, True):
        if on:
            P.warmstart_attach(net)
        P.set_point(m_lin)
        P.hessian_apply(Omega, out=Y)                           # warm-up (graphs, workspaces)
        ts, its = [], []
        for _ in range(3):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            st = P.hessian_apply(Omega, out=Y)[1]
            e1.record()
            e1.synchronize()
            ts.append(e0.elapsed_time(e1) / 1e3)
            its.append(st["iterations"])
        key = "learned" if on else "zero"
        out[f"pcg_iterations_{key}"] = statistics.median(its)
        out[f"actions_per_s_{key}"] = s / statistics.median(ts)
    c = P.warmstart_counts()
    # network inference alone, per column
    H, Wd = P.warmstart_grid()
    xin = torch.zeros((net.cap, 3, H, Wd), dtype=torch.float32, device=dev)
    net.forward(xin)
    fwd_ms = {}
    for tc in (True, False):  # the tensor-core convolutions (the default), then the FP32-pipe kernels
        net.tensor_cores = tc
        net.forward(xin)
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(3):
            net.forward(xin)
        e1.record()
        e1.synchronize()
        fwd_ms[tc] = e0.elapsed_time(e1) / 3 / net.cap
    P.warmstart_attach(None)
    P.set_point(m_lin)
    net.close()
    return {"train_samples": nsamp, "prior_draws": args.ws_draws, "epochs": args.ws_epochs,
            "generate_s": t_gen, "train_s": t_train, "loss_first_epoch": float(losses[0]),
            "loss_last_epoch": float(losses[-1]), **out, "guesses": c["guesses"], "fallbacks": c["fallbacks"],
            "forward_ms_per_column": fwd_ms[True], "forward_ms_per_column_fp32_pipes": fwd_ms[False],
            "note": ("same tolerance either way; the zero start stays the default of the timed step, "
                     "the learned start pays only if its inference costs less than the iterations it saves")}


def run_batch(args, rank, world):
    """64 uneven problems concurrently: MAP + k=30 eigenpairs for all, then one block of
    k+p = 40 Hessian actions per problem at its MAP (the timed step)."""
    import torch
    from paper_1909_03948_gb300 import Batch, algorithmic_bytes, kernel_launches
    torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", "0")))
    dev = torch.device("cuda", torch.cuda.current_device())
    ws = W.batch_workloads(seed=W.SEED_BASE + 3 + 1000 * rank)
    Ps = [synthetic_problem(w, dev, args.precision) for w in ws]
    if args.tuning:                       # fixed solver settings on every problem
        fixed = parse_tuning(args.tuning)
        for P in Ps:
            P.set_tuning(**fixed)
    Om = [torch.tensor(np.ascontiguousarray(W.omega(w).T), device=dev) for w in ws]
    B = Batch(Ps)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    ms, lams, Vs, nst = B.map_and_eig([P.zeros() for P in Ps], 30, 10, Om)
    torch.cuda.synchronize()
    t_me = time.perf_counter() - t0
    B.set_point(ms)
    for _ in range(max(args.warmup, 3)):
        B.hessian_apply(Om)
    flush = torch.empty(512 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    torch.cuda.synchronize()
    times = []
    l0 = kernel_launches()
    clocks = ClockSampler(torch.cuda.current_device())
    for _ in range(args.steps):
        flush.fill_(1.0)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        B.hessian_apply(Om)            # returns after every problem's stream has finished
        e1.record()
        e1.synchronize()
        times.append(e0.elapsed_time(e1) / 1e3)
    clk = clocks.stop()
    launches = kernel_launches() - l0
    units = sum(w.k + w.p for w in ws)
    value, t_total = weak_scaling_value(sum(times), args.steps * units, world, dev)
    # algorithmic bytes of one batch step, counted on a pass with profiling on (direct launches)
    for P in Ps:
        P.profile_enable(True)
    b0 = algorithmic_bytes()
    B.hessian_apply(Om)
    torch.cuda.synchronize()
    b1 = algorithmic_bytes()
    for P in Ps:
        P.profile_enable(False)
    step_bytes = {k: b1[k] - b0[k] for k in b0}
    tot = sum(step_bytes.values())
    ms_step = 1e3 * t_total / args.steps
    peak, src = measured_peak()
    roof = {"bound": "hbm", "achieved": tot / (ms_step * 1e-3) / 1e9, "peak": peak, "unit": "GB/s",
            "frac": tot / (ms_step * 1e-3) / 1e9 / peak, "traffic": None, "kernel": "whole batch step",
            "peak_source": src,
            "step": {"bytes_per_step": tot, "ms_per_step": ms_step,
                     "families": {k: {"bytes_per_step": v, "share_of_bytes": v / tot if tot else None}
                                  for k, v in step_bytes.items()},
                     "how": ("algorithmic bytes of every launch of one batch step (library counter, direct-launch "
                             "pass) over the timed steps' mean duration")}}
    # e2e: every problem's block copied from pinned host memory and the results read back
    Xh = [torch.empty(X.shape, dtype=torch.float64).pin_memory() for X in Om]
    for xh, X in zip(Xh, Om):
        xh.copy_(X.cpu())
    Yh = [torch.empty_like(x).pin_memory() for x in Xh]
    Xd = [torch.empty_like(X) for X in Om]
    e2e_times = []
    for _ in range(args.steps):
        flush.fill_(1.0)
        torch.cuda.synchronize()
        ta = time.perf_counter()
        for xd, xh in zip(Xd, Xh):
            xd.copy_(xh, non_blocking=True)
        torch.cuda.synchronize()      # the problems run on their own non-blocking streams
        Ys = B.hessian_apply(Xd)
        for yh, y in zip(Yh, Ys):
            yh.copy_(y, non_blocking=True)
        torch.cuda.synchronize()
        e2e_times.append(time.perf_counter() - ta)
    e2e_val = weak_scaling_value(sum(e2e_times), args.steps * units, world, dev)[0]
    io_bytes = sum(X.numel() * 8 for X in Om)
    # the same blocks one problem after another (no concurrency), for the per-problem rates
    alone = []
    for P, X in zip(Ps, Om):
        torch.cuda.synchronize()
        a = time.perf_counter()
        P.hessian_apply(X)
        torch.cuda.synchronize()
        alone.append(time.perf_counter() - a)
    B.close()
    if rank != 0:
        return
    cpu = None
    if not args.no_cpu and world == 1:
        try:
            val, sampled = oracle_batch_rate(ws)
            cpu = {"value": val, "unit": "actions/s", "cores": 1, "kind": "oracle",
                   "sample": f"{sampled} of {len(ws)} problems (every 8th): one K(m) factorisation and one column "
                             f"each, extrapolated to 40-column blocks and to the whole batch, 1 thread"}
        except Exception as ex:  # pragma: no cover
            cpu = {"value": None, "unit": "actions/s", "cores": 1, "kind": "oracle", "sample": f"failed: {ex}"}
    line = {
        "metric": METRIC, "value": value, "unit": "actions/s", "n_gpus": world, "steps": args.steps,
        "warmup": max(args.warmup, 3), "ms_per_step": 1e3 * t_total / args.steps, "higher_is_better": True,
        "scaling": "weak", "vs_baseline": None, "dtype": "f32-in-f64-IR", "data": "synthetic",
        "config": {"workload": f"batch64: {len(ws)} independent 2D problems, N log-uniform in [64, 512] "
                               f"(multiples of 32), q in [100, 800], one block of k+p=40 GN Hessian actions per "
                               f"problem at its MAP, problems concurrent on per-problem streams",
                   "l2": "flushed (512 MB write) before every timed step"},
        "gpu_launches": launches, "clocks": clk, "build": build_record(),
        "e2e": {"value": e2e_val, "unit": "actions/s", "h2d_bytes_per_step": io_bytes, "d2h_bytes_per_step": io_bytes},
        "roofline": roof, "cpu_baseline": cpu,
        "time_to_map_eig_s": t_me,
        "map_eig_actions_per_s": sum(x["cg_iterations"] + 2 * 40 for x in nst) / t_me,
        "sequential_seconds_per_step": sum(alone), "concurrency_speedup": sum(alone) / (t_total / args.steps),
        "per_problem": [{"N": w.N, "q": w.nobs, "newton_iterations": x["iterations"], "alone_actions_per_s": 40 / a}
                        for w, x, a in zip(ws, nst, alone)],
    }
    print(json.dumps(line), flush=True)


def main():
    args = parse()
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    if args.impl == "reference":
        run_reference(args, rank, world)
        return
    if world > 1:
        import torch
        import torch.distributed as dist
        torch.cuda.set_device(int(os.environ.get("LOCAL_RANK", "0")))
        dist.init_process_group("nccl")
    if args.workload == "batch64":
        run_batch(args, rank, world)
    else:
        run_ours(args, rank, world)
    if world > 1:
        import torch.distributed as dist
        dist.barrier()
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
