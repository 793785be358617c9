"""Benchmark: k-point eigenpairs/s of the Bloch-wave band solve on one GB300.

Workload (default): 128^3 periodic cell, 200 Voronoi grains, Cu-like cubic
stiffness with a <001> von Mises-Fisher fibre (kappa 20), 10 bands at 64
wave vectors on Gamma-X-M-Gamma-R; synthetic, seeded.  A step solves one
batch of wave vectors of that path (--k-per-step) to the frequency accuracy
of the form (chosen: FP32 fields + FP64 refinement; plain: FP64 throughout).

Prints one JSON line (rank 0).  Under torchrun each rank solves its own k
batches (no collective on the data path; barrier + max over ranks for time).
"""
from __future__ import annotations

import argparse
import json
import math
import os
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "k-point eigenpairs/s at 128^3 (freq rel err <=1e-6)"


def metric_of(grid):
    """The headline metric's name for a workload grid (the default workload is 128^3)."""
    if tuple(grid) == (128, 128, 128):
        return METRIC
    g = "x".join(str(int(v)) for v in grid) if len(set(grid)) > 1 else f"{int(grid[0])}^3"
    return f"k-point eigenpairs/s at {g} (freq rel err <=1e-6)"
PEAKS_FILE = os.path.join(ROOT, "MEASURED_PEAKS.json")
FALLBACK_HBM = 6800.0
KAPPLY_BYTES_PER_VOXEL = {1: 436.0, 0: 868.0, 2: 868.0}   # algorithmic bytes per voxel, 5-pass chain (FF: 16 B complex)
# DRAM bytes (dram__bytes_read.sum + dram__bytes_write.sum over the five passes) per system of the
# FP32 fast-pass K-apply at 128^3, from one ncu capture of a 4-system launch (1832.1 MB read +
# 1521.4 MB written); it scales with the systems per launch.  Valid only while the pass sources hash
# to `sources_sha256` (fpasses.cuh, fft.cuh, common.cuh in that order); otherwise traffic is null.
KAPPLY_TRAFFIC = {"grid": (128, 128, 128), "precision": 1, "fft_variant": 0,
                  "bytes_per_system": 3353.47e6 / 4,
                  "sources_sha256": "f06f136dd1beb7cb1c707d9ef2f210dcea2edd7644760771e2ab5efd5df95a20"}


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=2)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="rve128_g200")
    ap.add_argument("--form", default="chosen", choices=["chosen", "chosen-subspace", "lobpcg", "plain"])
    ap.add_argument("--k-per-step", type=int, default=8)
    ap.add_argument("--no-e2e", action="store_true")
    ap.add_argument("--no-cpu", action="store_true")
    ap.add_argument("--no-path", action="store_true",
                    help="skip the leg that solves the whole 64-point path in one bloch_solve_bands call")
    ap.add_argument("--no-plain", action="store_true",
                    help="skip the leg that times the plain FP64 cuFFT form on two 4-point batches")
    ap.add_argument("--max-outer", type=int, default=100, help="sweep cap (profiling runs bound it)")
    ap.add_argument("--kapply-only", action="store_true", help="time only the K-apply chain")
    ap.add_argument("--kapply-nb", type=int, default=0, help="systems per K-apply launch (0 = block size)")
    ap.add_argument("--alu-peaks", action="store_true",
                    help="measure FP64/FP32 FMA throughput and time the FP64, float-float and FP32 operator chains "
                         "on --kapply-nb systems against it")
    ap.add_argument("--wave-speeds", action="store_true",
                    help="low-frequency wave speeds (Section 5.2, Eq. wave_speed2) of the workload along x, y "
                         "and z: Hellmann-Feynman slopes of the three acoustic branches at k = K d, FP64 form")
    ap.add_argument("--props", action="store_true",
                    help="time the band-property calls (group velocity, real-space fields with strain) on "
                         "--kapply-nb vectors (default 10) against one K-apply of the same vectors")
    ap.add_argument("--pcg-only", type=int, default=0, metavar="ITERS",
                    help="time only ITERS FP32 PCG iterations on --kapply-nb systems (default 4)")
    ap.add_argument("--kapply-prec", default="form", choices=["form", "fp32", "fp64", "ff"],
                    help="with --kapply-only: precision of the timed chain (form = the form's), with --fft-variant "
                         "taken as given")
    ap.add_argument("--fft-variant", type=int, default=0, choices=[0, 1, 2],
                    help="0: two-stage register FFT passes, 1: mixed-radix passes everywhere, 2: cuFFT baseline")
    ap.add_argument("--precond", default="green", choices=["green", "learned"],
                    help="green: the Green operator P^-1 (the paper); learned: train the learned Fourier-space "
                         "preconditioner first (untimed, reported under 'precond') and solve with it")
    ap.add_argument("--lp-cells", type=int, default=16, help="training cells (64^3 Zener family) for --precond learned")
    ap.add_argument("--lp-steps", type=int, default=500, help="Adam steps for --precond learned")
    ap.add_argument("--learned-config4", action="store_true",
                    help="the learned-preconditioner study at its configured scale: train on --lp-cells seeded 64^3 "
                         "Zener cells (400 for the study), then on a 128^3, 300-grain test cell report PCG iterations "
                         "at equal tolerance and chosen-form eigenpairs/s with the Green and the learned operator")
    ap.add_argument("--no-trace", action="store_true",
                    help="skip the extra traced (untimed) step that reports the solver's phase breakdown")
    ap.add_argument("--tensor-gram", type=int, default=0, choices=[0, 1],
                    help="1: Algorithm 1 projections of FP32 blocks on the tensor cores (tcgen05)")
    ap.add_argument("--ncv", type=int, default=0, help="Lanczos basis size of the chosen form (0: max(2n+1, 20))")
    ap.add_argument("--k-batch", type=int, default=0,
                    help="wave vectors advanced together by the chosen form (0: the library's choice, 8)")
    ap.add_argument("--hybrid-tol", type=float, default=0.0,
                    help="Lanczos-stage hand-over tolerance of the chosen form (0: max(1e-5, 10 tol_eig))")
    ap.add_argument("--refine-arith", type=int, default=1, choices=[0, 1],
                    help="arithmetic of the chosen form's FP64 check: 0 IEEE FP64, 1 float-float operator "
                         "applies with FP64 sums")
    ap.add_argument("--cuda-graph", type=int, default=1, choices=[0, 1],
                    help="1: PCG loop as one CUDA graph with a device-side while node; 0: host-driven loop "
                         "(same kernels; used for per-launch profiling)")
    return ap.parse_args()


def dist_init(args):
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    if ws > 1:
        import torch
        import torch.distributed as dist
        if args.impl == "ours":
            torch.cuda.set_device(local)
            dist.init_process_group("nccl")
        else:
            dist.init_process_group("gloo")
    return ws, rank, local


def k_indices(step, rank, ws, kps, nk):
    """Wave-vector indices solved by `rank` at `step`: the ranks of one step
    take disjoint consecutive batches of the path (weak scaling, no data-path
    collective)."""
    return [((step * ws + rank) * kps + i) % nk for i in range(kps)]


def barrier(ws):
    if ws > 1:
        import torch.distributed as dist
        dist.barrier()


def max_over_ranks(ws, v):
    if ws == 1:
        return v
    import torch
    import torch.distributed as dist
    t = torch.tensor([v], dtype=torch.float64, device="cuda" if torch.cuda.is_available() else "cpu")
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


class ClockSampler:
    """nvidia-smi clocks and throttle reasons sampled during the timed region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
         "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
         "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
            out, _ = self.proc.communicate()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.strip().splitlines():
            f = [x.strip() for x in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for nm, val in zip(names, f[5:9]):
                if val.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": float(np.median(sm)) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def peaks():
    try:
        with open(PEAKS_FILE) as f:
            d = json.load(f)
        return float(d["hbm_gbs"]), "measured"
    except Exception:
        return FALLBACK_HBM, "fallback"


def oracle_sample(p, n_iter=2):
    """Oracle as it stands, timed on a bounded sample: n_iter PCG iterations of
    Algorithm 2 at the workload's grid for its first non-zero wave vector.
    Returns (seconds per operator apply, threads it kept busy = process CPU
    time / wall time, rounded, at least 1)."""
    from oracle import bloch_oracle as O
    from paper_2106_12487_gb300 import synth
    med = O.Medium.from_problem(p)
    k = p.k_list[1]
    b = synth.random_field(p.grid, 99)
    t0, c0 = time.perf_counter(), time.process_time()
    O.pcg(lambda x: O.apply_K(med, k, x), lambda x: O.apply_precond(med, k, x), b, 1e-30, n_iter)
    dt, dc = time.perf_counter() - t0, time.process_time() - c0
    # pcg runs n_iter operator applies plus one for the final true residual
    return dt / (n_iter + 1), max(1, int(round(dc / max(dt, 1e-9))))


def oracle_applies_per_eigenpair():
    """K-applies per eigenpair of the oracle's own band solve (shift-invert
    Lanczos, ARPACK) on the 16^3 workload, as recorded by
    tests/golden/make_golden.py."""
    path = os.path.join(ROOT, "tests", "golden", "rve16_g8_bands.json")
    with open(path) as f:
        g = json.load(f)
    return float(g["oracle_cg_iters"]) / float(g["eigenpairs"]), "rve16_g8 oracle Lanczos"


def _oracle_k_solve(task):
    """Worker of the oracle baseline (spawned process): the oracle's band solve
    (shift-invert Lanczos through ARPACK, Algorithm 2 PCG) of one wave vector
    of a workload.  Returns (omega, wall s, process CPU s)."""
    name, i, tol = task
    from oracle import bloch_oracle as O
    from paper_2106_12487_gb300 import synth
    p = synth.workload(name)
    med = O.Medium.from_problem(p)
    t0, c0 = time.perf_counter(), time.process_time()
    res = O.solve_bands(med, p.k_list[i:i + 1], p.n_bands, tol, tol, method="lanczos")
    return res.omega[0].tolist(), time.perf_counter() - t0, time.process_time() - c0


def _noop(_):
    return 0


def oracle_band_baseline(name="rve16_g8", tol=1e-10, one_core_k=5):
    """The FP64 oracle as it stands, measured (not extrapolated) on a whole
    small workload: every wave vector of `name` solved in a spawned process
    pool over the host cores (one wave vector per process, one thread each),
    plus one wave vector alone on one core.  Returns the two rates in
    eigenpairs/s, the cores kept busy and the oracle's frequencies."""
    import multiprocessing as mp
    from paper_2106_12487_gb300 import synth
    p = synth.workload(name)
    nk = int(p.k_list.shape[0])
    saved = {v: os.environ.get(v) for v in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS")}
    for v in saved:
        os.environ[v] = "1"
    try:
        nproc = max(1, min(nk, os.cpu_count() or 1))
        ctx = mp.get_context("spawn")
        with ctx.Pool(nproc) as pool:
            pool.map(_noop, range(nproc))          # interpreters started before the clock
            t0 = time.perf_counter()
            res = pool.map(_oracle_k_solve, [(name, i, tol) for i in range(nk)], chunksize=1)
            wall = time.perf_counter() - t0
            one = pool.apply(_oracle_k_solve, ((name, one_core_k, tol),))
    finally:
        for v, old in saved.items():
            if old is None:
                os.environ.pop(v, None)
            else:
                os.environ[v] = old
    cpu = sum(r[2] for r in res)
    omega = np.array([r[0] for r in res])
    return {"workload": name, "grid": list(p.grid), "n_k": nk, "n_bands": int(p.n_bands), "tol": tol,
            "all_cores": {"value": nk * p.n_bands / wall, "wall_s": wall, "processes": nproc,
                          "cores": max(1, int(round(cpu / max(wall, 1e-9))))},
            "one_core": {"value": p.n_bands / one[1], "wall_s": one[1], "k_index": one_core_k, "cores": 1},
            "omega": omega}


def gpu_band_same_config(name, omega_ref):
    """Our band solve on the oracle-baseline workload, all its wave vectors in
    one bloch_solve_bands call per form (FP64 plain form with our passes at the
    oracle's tolerance; FP32 chosen form), CUDA events after one warm-up call;
    max relative frequency difference to the oracle's."""
    import torch
    from paper_2106_12487_gb300 import bloch, synth
    p = synth.workload(name)
    out = {}
    forms = {"fp64_plain": dict(precision=bloch.FP64, method=bloch.LANCZOS, tol_lin=1e-10, tol_eig=1e-10),
             "chosen": dict(precision=bloch.FP32, method=bloch.LANCZOS, tol_lin=1e-2, tol_eig=1e-5,
                            block=p.n_bands + 2, max_cg=500, refine_arith=1)}
    stream = torch.cuda.current_stream()
    for form, opt in forms.items():
        plan = bloch.Plan.from_problem(p, **opt)
        plan.solve_bands(p.k_list, p.n_bands, allow_nonconv=True)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record(stream)
        om, st, status = plan.solve_bands(p.k_list, p.n_bands, allow_nonconv=True)
        e1.record(stream)
        torch.cuda.synchronize()
        dt = e0.elapsed_time(e1) / 1000.0
        nz = omega_ref > 0
        out[form] = {"value": p.k_list.shape[0] * p.n_bands / dt, "status": int(status),
                     "max_rel_freq_diff_vs_oracle": float(np.max(np.abs(om[nz] / omega_ref[nz] - 1.0)))}
        plan.close()
    return out


def run_reference(args, ws, rank):
    """The oracle (FP64 numpy) on the host cores, same workload and metric."""
    if rank != 0:
        return
    from paper_2106_12487_gb300 import synth
    p = synth.workload(args.workload)
    a_per_pair, src = oracle_applies_per_eigenpair()
    for _ in range(args.warmup):
        oracle_sample(p, 1)
    t_apply, threads = [], []
    t0 = time.perf_counter()
    for _ in range(args.steps):
        ta_s, th = oracle_sample(p, 1)
        t_apply.append(ta_s)
        threads.append(th)
    wall = time.perf_counter() - t0
    ta = float(np.mean(t_apply))
    value = 1.0 / (ta * a_per_pair)
    sample = (f"estimate, not a measured band solve: {args.steps} x (1 PCG iteration + residual check) of the "
              f"FP64 oracle at {p.grid} ({ta:.2f} s per A_k apply, measured); eigenpairs/s = 1/(s per apply x "
              f"{a_per_pair:.1f} applies per eigenpair, {src}); a 128^3 band solve of the oracle takes hours")
    line = {"impl": "reference", "metric": metric_of(p.grid), "value": value, "unit": "eigenpairs/s", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1000.0 * wall / max(args.steps, 1),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": {"workload": args.workload, "grid": list(p.grid),
                                            "n_bands": p.n_bands, "n_k": int(p.k_list.shape[0])},
            "cpu_baseline": {"value": value, "unit": "eigenpairs/s", "cores": max(threads) if threads else 1,
                             "kind": "oracle",
                             "sample": sample},
            "e2e": {"value": value, "unit": "eigenpairs/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def kapply_traffic(p, prec, fft_variant, q):
    """Measured DRAM bytes per launch of q systems, or None when no capture
    covers this kernel build and workload."""
    import hashlib
    t = KAPPLY_TRAFFIC
    if tuple(p.grid) != t["grid"] or prec != t["precision"] or fft_variant != t["fft_variant"]:
        return None
    h = hashlib.sha256()
    for f in ("fpasses.cuh", "fft.cuh", "common.cuh"):
        with open(os.path.join(ROOT, "paper_2106_12487_gb300", "csrc", f), "rb") as fh:
            h.update(fh.read())
    if h.hexdigest() != t["sources_sha256"]:
        return None
    return t["bytes_per_system"] * q


def kapply_roofline(plan, p, prec, nb=0, fft_variant=0):
    """The dominant kernel chain: the 5-pass K-apply on a block of nb systems
    (default: one subspace block), timed with CUDA events on the launching
    stream after warm-up; inputs (nb x 3 x V complex) and the 6-component
    intermediates are larger than L2 at 128^3."""
    import torch
    from paper_2106_12487_gb300 import bloch
    q = nb if nb > 0 else min(2 * p.n_bands, p.n_bands + 8)
    dt = torch.complex64 if prec == bloch.FP32 else torch.complex128
    u = torch.randn(q * 3 * plan.V, dtype=dt, device="cuda")
    out = torch.empty_like(u)
    kq = np.repeat(p.k_list[5:6], q, axis=0)
    stream = torch.cuda.current_stream()
    for _ in range(3):
        plan.apply_K(kq, u, out, precision=prec)
    torch.cuda.synchronize()
    reps = 10
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(reps):
        plan.apply_K(kq, u, out, precision=prec)
    e1.record(stream)
    torch.cuda.synchronize()
    t_apply = e0.elapsed_time(e1) / 1000.0 / reps
    alg_bytes = KAPPLY_BYTES_PER_VOXEL[prec] * plan.V * q
    peak, peak_src = peaks()
    achieved = alg_bytes / t_apply / 1e9
    return {"bound": "hbm", "achieved": achieved, "peak": peak, "unit": "GB/s", "frac": achieved / peak,
            "traffic": kapply_traffic(p, prec, fft_variant, q), "kernel": f"K-apply 5-pass chain, {q} systems at {tuple(p.grid)} ({peak_src} peak)",
            "ms_per_launch": t_apply * 1000.0, "alg_bytes_per_launch": alg_bytes}


def kapply_flops_per_voxel(grid):
    """Algorithmic flops of one A_k apply per voxel: 36 length-N complex
    transforms per voxel (6 along z, 6 along y, 12 along x, 6 along y, 6 along
    z) at 5 log2(N) flops per point each, plus the pointwise strain (24),
    stress (a real 6x6 on a complex 6-vector, 144) and divergence (30)."""
    import math
    nx, ny, nz = grid
    return 5.0 * (12 * math.log2(nz) + 12 * math.log2(ny) + 12 * math.log2(nx)) + 24 + 144 + 30


def props_leg(plan, p, nb):
    """Group velocity (Eq. c_group) and real-space eigenvector fields with
    strain (Eq. rotate_eigenvector) of nb vectors, CUDA events after one
    warm-up call each, next to one K-apply of the same vectors."""
    import torch
    from paper_2106_12487_gb300 import bloch
    prec = plan.precision
    dt = torch.complex64 if prec == bloch.FP32 else torch.complex128
    g = torch.Generator(device="cuda").manual_seed(0)
    u = torch.randn(nb * 3 * plan.V, dtype=dt, device="cuda", generator=g)
    ur = torch.empty_like(u)
    eps = torch.empty(nb * 6 * plan.V, dtype=dt, device="cuda")
    kq = np.repeat(p.k_list[5:6], nb, axis=0)
    stream = torch.cuda.current_stream()

    def timed(fn):
        fn()
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        fn()
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1)

    t_k = timed(lambda: plan.apply_K(kq, u, ur))
    t_gv = timed(lambda: plan.group_velocity(kq, u))
    t_ev = timed(lambda: plan.eigvec_real(u, ur, eps))
    return {"vectors": nb, "grid": list(p.grid), "ms_apply_K": t_k, "ms_group_velocity": t_gv,
            "ms_eigvec_real_with_strain": t_ev, "group_velocity_over_apply_K": t_gv / t_k,
            "eigvec_real_over_apply_K": t_ev / t_k}


def voigt_christoffel_speeds(p, d):
    """Plane-wave speeds along d of the volume-average (Voigt) stiffness and
    density of the cell: sqrt of the eigenvalues (ascending) of the Christoffel
    matrix C0_ijkl d_j d_l / rho_bar."""
    ids = np.asarray(p.grain_ids).ravel()
    counts = np.bincount(ids, minlength=len(p.rho)) / ids.size
    C0 = np.einsum("g,gij->ij", counts, np.asarray(p.C_per_grain, float))
    rho = float(np.dot(counts, p.rho))
    vi = ((0, 5, 4), (5, 1, 3), (4, 3, 2))   # Voigt index of the tensor pair (i, j)
    C4 = np.array([[[[C0[vi[i][j], vi[k][l]] for l in range(3)] for k in range(3)] for j in range(3)]
                   for i in range(3)])
    d = np.asarray(d, float) / np.linalg.norm(d)
    return np.sqrt(np.linalg.eigvalsh(np.einsum("ijkl,j,l->ik", C4, d, d) / rho))


def wave_speeds_leg(p, K_frac=0.01):
    """Wave speeds along x, y, z (Eq. wave_speed2): the three lowest bands at
    k = K d (K = K_frac pi / L) from bloch_solve_bands (FP64 plain form's
    precision and tolerances, our passes), their group velocities from
    bloch_group_velocity, projected on d.  Next to them, the Christoffel speeds
    of the volume-average stiffness C0 (Eq. wave_speed with the Voigt average in
    place of the paper's FFT-homogenised C, an upper bound)."""
    import torch
    from paper_2106_12487_gb300 import bloch
    plan = bloch.Plan.from_problem(p, precision=bloch.FP64, method=bloch.LANCZOS, tol_lin=1e-10,
                                   tol_eig=1e-10, max_cg=2000)
    out = {}
    for name, d in (("x", (1.0, 0.0, 0.0)), ("y", (0.0, 1.0, 0.0)), ("z", (0.0, 0.0, 1.0))):
        d = np.array(d)
        K = K_frac * math.pi / p.L[int(np.argmax(d))]
        vecs = torch.zeros(3 * 3 * plan.V, dtype=torch.complex128, device="cuda")
        omega, _, st = plan.solve_bands((K * d)[None], 3, vecs_out=vecs)
        _, c = plan.group_velocity(np.repeat((K * d)[None], 3, 0), vecs)
        out[name] = {"speeds": (c @ d).tolist(), "secant": (omega[0] / K).tolist(), "status": int(st),
                     "voigt_christoffel": voigt_christoffel_speeds(p, d).tolist()}
    plan.close()
    return {"workload": p.name if hasattr(p, "name") else None, "K_frac_pi_over_L": K_frac, "directions": out}


def alu_peaks_leg(p, opt, nb):
    """FMA peaks of the device and the operator chains timed against them."""
    from paper_2106_12487_gb300 import bloch
    g64, g32 = bloch.fma_peaks()
    fpv = kapply_flops_per_voxel(p.grid)
    out = {"fma_peaks": {"fp64_gflops": g64, "fp32_gflops": g32, "how": "bloch_fma_peaks: CUDA events, "
                         "8 x 256-thread CTAs per SM of independent FMA chains, FMA = 2 flops"},
           "flops_per_voxel": fpv, "systems": nb, "chains": {}}
    for name, prec in (("fp64", bloch.FP64), ("ff", bloch.FF), ("fp32", bloch.FP32)):
        plan = bloch.Plan.from_problem(p, **dict(opt, precision=bloch.FP32 if prec == bloch.FP32 else bloch.FP64,
                                                 fft_variant=0))
        r = kapply_roofline(plan, p, prec, nb, 0)
        plan.close()
        gf = fpv * plan.V * nb / (r["ms_per_launch"] * 1e-3) / 1e9
        out["chains"][name] = {"ms_per_launch": r["ms_per_launch"], "gflops": gf,
                               "frac_of_fp64_fma_peak": gf / g64, "frac_of_fp32_fma_peak": gf / g32,
                               "hbm_frac": r["frac"]}
    return out


# FP32, c = 8 B, per voxel, system and iteration.  Plain-form baseline (fft_variant 2): K-apply
# 54c + 4, k_cg_update 9c, k_cg_pupdate 15c.
PCG_BYTES_PER_VOXEL = 628.0
# The pass chain: passes 1-4 (9 + 12 + 12 + 12)c + 4, the divergence pass that updates r in place of
# storing Ap 6c + 3c + 3c, k_cg_pupdate 15c.
PCG_CHAIN_BYTES_PER_VOXEL = 580.0


def pcg_bytes_per_voxel(fft_variant):
    """Algorithmic bytes of one FP32 PCG iteration per voxel and system."""
    return PCG_BYTES_PER_VOXEL if fft_variant == 2 else PCG_CHAIN_BYTES_PER_VOXEL


def pcg_roofline(plan, p, nb, iters):
    """One FP32 PCG iteration (Algorithm 2) on nb systems: `iters` iterations
    with a tolerance no system reaches, timed with CUDA events on the
    launching stream after one warm-up solve; the time per iteration includes
    the loop's control (graph conditional node or host loop)."""
    import torch
    from paper_2106_12487_gb300 import bloch
    g = torch.Generator(device="cuda").manual_seed(0)
    b = torch.randn(nb * 3 * plan.V, dtype=torch.complex64, device="cuda", generator=g)
    x = torch.zeros_like(b)
    kq = np.repeat(p.k_list[5:6], nb, axis=0)
    stream = torch.cuda.current_stream()
    plan.pcg(kq, b, x, 1e-30, max_iter=iters, precision=bloch.FP32, allow_nonconv=True)
    torch.cuda.synchronize()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    it, _, _ = plan.pcg(kq, b, x, 1e-30, max_iter=iters, precision=bloch.FP32, allow_nonconv=True)
    e1.record(stream)
    torch.cuda.synchronize()
    n_it = int(it.max())
    t_it = e0.elapsed_time(e1) / 1000.0 / max(n_it, 1)
    alg = pcg_bytes_per_voxel(plan.options.fft_variant) * plan.V * nb
    peak, peak_src = peaks()
    return {"bound": "hbm", "achieved": alg / t_it / 1e9, "peak": peak, "unit": "GB/s",
            "frac": alg / t_it / 1e9 / peak, "kernel": f"FP32 PCG iteration, {nb} systems at {tuple(p.grid)} "
            f"({peak_src} peak)", "iterations": n_it, "ms_per_iteration": t_it * 1000.0,
            "alg_bytes_per_iteration": alg}


def train_learned(args):
    """Learned Fourier-space preconditioner: record CG pairs on 64^3 cells of
    the Zener family (two wave vectors each), then full-batch Adam.  Untimed;
    returns the network and what the JSON line reports about it."""
    import torch
    from paper_2106_12487_gb300 import bloch, synth
    t0 = time.perf_counter()
    lp = bloch.LearnedPrecond(seed=7)
    for i in range(args.lp_cells):
        c = synth.zener_cell((64, 64, 64), i)
        pl = bloch.Plan.from_problem(c, precision=bloch.FP32)
        pick = np.random.default_rng(31 + i).choice(len(c.k_list) - 1, 2, replace=False) + 1
        lp.collect(pl, c.k_list[pick], n_rhs=2, n_iters=12, seed=31 + i)
        pl.close()
    L0, _ = lp.loss_grad()
    lp.train(args.lp_steps, lr=3e-3)
    L1, _ = lp.loss_grad()
    torch.cuda.synchronize()
    return lp, {"kind": "learned", "train_cells": args.lp_cells, "cell": [64, 64, 64], "adam_steps": args.lp_steps,
                "loss": [L0, L1], "train_s": time.perf_counter() - t0}


def learned_config4(args):
    """Learned preconditioner at the study's scale (one JSON line).  Training
    data: per cell, two wave vectors of its path and two seeded right-hand
    sides, 12 recorded PCG iterates each.  Test cell: 128^3, 300 Voronoi grains
    (seed 4), Haar orientations (seed 104), cubic with Zener ratio 2.5 (the
    middle of the training range)."""
    import torch
    from paper_2106_12487_gb300 import bloch, synth
    lp, info = train_learned(args)
    C11, C12 = synth.CU_CUBIC["C11"], synth.CU_CUBIC["C12"]
    C6 = synth.cubic_voigt(C11, C12, 2.5 * (C11 - C12) / 2)
    p = synth.polycrystal("config4_test", (128, 128, 128), 300, 4, 104, C6, synth.CU_CUBIC["rho"],
                          synth.kpath("GXMGR", 64), 10, 1e-10)
    out = {"study": "learned preconditioner, train 64^3 Zener cells, test 128^3 / 300 grains", "train": info}
    # PCG iterations at equal tolerance, 4 wave vectors x 4 right-hand sides
    kidx = [5, 20, 36, 50]
    iters = {}
    for name, use in (("green", False), ("learned", True)):
        plan = bloch.Plan.from_problem(p, precision=bloch.FP32, cuda_graph=1)
        if use:
            bloch.set_preconditioner(plan, lp)
        for tol in (1e-2, 1e-5):
            tot = []
            for j, ki in enumerate(kidx):
                b = torch.from_numpy(synth.random_field(p.grid, 300 + j, batch=4) * 1e18).to(
                    device="cuda", dtype=torch.complex64)
                x = torch.zeros_like(b)
                it, rel, _ = plan.pcg(np.repeat(p.k_list[ki:ki + 1], 4, 0), b, x, tol, 3000, allow_nonconv=True)
                tot.extend(int(v) for v in it)
            iters.setdefault(name, {})[str(tol)] = {"mean": float(np.mean(tot)), "all": tot}
        plan.close()
    out["pcg_iterations"] = iters
    # chosen-form band solve of 8 wave vectors (after one warm-up batch), both operators
    opt = dict(precision=bloch.FP32, method=bloch.LANCZOS, tol_lin=1e-2, tol_eig=1e-5, max_cg=500,
               block=p.n_bands + 2, max_outer=args.max_outer, refine_arith=args.refine_arith)
    stream = torch.cuda.current_stream()
    om_ref = None
    for name, use in (("green", False), ("learned", True)):
        plan = bloch.Plan.from_problem(p, **opt)
        if use:
            bloch.set_preconditioner(plan, lp)
        plan.solve_bands(p.k_list[0:8], p.n_bands, allow_nonconv=True)
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record(stream)
        om, st, status = plan.solve_bands(p.k_list[8:16], p.n_bands, allow_nonconv=True)
        e1.record(stream)
        torch.cuda.synchronize()
        dt = e0.elapsed_time(e1) / 1000.0
        out.setdefault("band_solve", {})[name] = {"eigenpairs_per_s": 8 * p.n_bands / dt, "status": int(status),
                                                  "cg_iterations": st["cg_iterations"]}
        if om_ref is None:
            om_ref = om
        else:
            out["band_solve"]["max_rel_freq_diff"] = float(np.max(np.abs(om / om_ref - 1.0)))
        plan.close()
    print(json.dumps(out), flush=True)


def run_ours(args, ws, rank, local):
    import torch
    from paper_2106_12487_gb300 import bloch, synth

    if not torch.cuda.is_available():
        raise SystemExit("bench.py needs a CUDA device")
    torch.cuda.set_device(local)
    if args.learned_config4:
        learned_config4(args)
        return
    p = synth.workload(args.workload)
    prec = bloch.FP64 if args.form == "plain" else bloch.FP32
    if args.form == "chosen":
        # FP32 fields and PCG: FP32 shift-invert Lanczos, then Algorithm 1 refinement
        # sweeps with the FP64 residual check.  The refinement (residual-correction
        # form) fixes the final accuracy, so the inner PCG tolerance of both stages
        # only trades PCG iterations against sweeps: 1e-2 was fastest at equal
        # frequencies (relative change <= 1e-10 against 1e-5 inner solves)
        # Block n + 2 for the refinement: the Lanczos stage hands over good vectors,
        # so two guard vectors suffice (12 was fastest of 12-18 at equal frequencies)
        opt = dict(precision=prec, method=bloch.LANCZOS, tol_lin=1e-2, tol_eig=1e-5, max_cg=500, block=p.n_bands + 2,
                   max_outer=args.max_outer, fft_variant=args.fft_variant, cuda_graph=args.cuda_graph,
                   tensor_gram=args.tensor_gram, ncv=args.ncv, hybrid_tol=args.hybrid_tol,
                   refine_arith=args.refine_arith, k_batch=args.k_batch)
    elif args.form == "lobpcg":
        # FP32 LOBPCG with the Green preconditioner (no inner PCG), FP64 residual check
        opt = dict(precision=prec, method=bloch.LOBPCG, tol_lin=1e-2, tol_eig=1e-5, max_cg=500, block=p.n_bands + 2,
                   max_outer=max(args.max_outer, 300), fft_variant=args.fft_variant, cuda_graph=args.cuda_graph)
    elif args.form == "chosen-subspace":
        # FP32 fields and PCG, subspace iteration with warm starts, FP64 residual check
        opt = dict(precision=prec, method=bloch.SUBSPACE, tol_lin=1e-3, tol_eig=1e-6, max_cg=500,
                   max_outer=args.max_outer, fft_variant=args.fft_variant, cuda_graph=args.cuda_graph,
                   tensor_gram=args.tensor_gram)
    else:
        # the paper's plain form: FP64, shift-invert Lanczos, cuFFT operator
        opt = dict(precision=prec, method=bloch.LANCZOS, tol_lin=1e-10, tol_eig=1e-10, max_cg=2000,
                   max_outer=args.max_outer, fft_variant=2 if args.fft_variant == 0 else args.fft_variant,
                   cuda_graph=args.cuda_graph)
    plan = bloch.Plan.from_problem(p, **opt)
    lp, lp_info = None, {"kind": "green"}
    if args.precond == "learned":
        lp, lp_info = train_learned(args)
        bloch.set_preconditioner(plan, lp)
    if args.alu_peaks:
        plan.close()
        leg = alu_peaks_leg(p, opt, args.kapply_nb or 4)
        if rank == 0:
            print(json.dumps({"alu": leg}), flush=True)
        return
    if args.wave_speeds:
        plan.close()
        leg = wave_speeds_leg(p)
        if rank == 0:
            print(json.dumps({"wave_speeds": leg}), flush=True)
        return
    if args.props:
        leg = props_leg(plan, p, args.kapply_nb or 10)
        if rank == 0:
            print(json.dumps({"props": leg}), flush=True)
        plan.close()
        return
    if args.pcg_only:
        roof = pcg_roofline(plan, p, args.kapply_nb or 4, args.pcg_only)
        if rank == 0:
            print(json.dumps({"pcg": roof}), flush=True)
        plan.close()
        return
    if args.kapply_only:
        if args.kapply_prec != "form":
            plan.close()
            prec = {"fp64": bloch.FP64, "fp32": bloch.FP32, "ff": bloch.FF}[args.kapply_prec]
            opt = dict(opt, precision=bloch.FP64 if prec == bloch.FF else prec, fft_variant=args.fft_variant)
            plan = bloch.Plan.from_problem(p, **opt)
        roof = kapply_roofline(plan, p, prec, args.kapply_nb, opt["fft_variant"])
        if rank == 0:
            print(json.dumps({"kapply": roof}), flush=True)
        plan.close()
        return
    nk = p.k_list.shape[0]
    kps = args.k_per_step

    def kbatch(step):
        return p.k_list[k_indices(step, rank, ws, kps, nk)]

    stream = torch.cuda.current_stream()
    for s in range(args.warmup):
        plan.solve_bands(kbatch(s), p.n_bands, allow_nonconv=True)
    torch.cuda.synchronize()
    clocks = ClockSampler(local)
    clocks.start()
    barrier(ws)
    torch.cuda.synchronize()
    ev0 = torch.cuda.Event(enable_timing=True)
    ev1 = torch.cuda.Event(enable_timing=True)
    stats_all, status_all = [], []
    launches0 = plan.kernel_launches
    ev0.record(stream)
    for s in range(args.steps):
        _, st, status = plan.solve_bands(kbatch(args.warmup + s), p.n_bands, allow_nonconv=True)
        stats_all.append(st)
        status_all.append(int(status))
    ev1.record(stream)
    torch.cuda.synchronize()
    barrier(ws)
    clk = clocks.stop()
    launches = plan.kernel_launches - launches0
    t = ev0.elapsed_time(ev1) / 1000.0
    t = max_over_ranks(ws, t)
    pairs = args.steps * kps * p.n_bands * ws
    value = pairs / t
    cg = sum(s["cg_iterations"] for s in stats_all)
    kap = sum(s["k_applies"] for s in stats_all)
    k_unconv = int(sum(s["k_unconverged"] for s in stats_all))
    covered = sorted({i for s in range(args.steps) for i in k_indices(args.warmup + s, rank, ws, kps, nk)})

    roof = kapply_roofline(plan, p, prec, args.kapply_nb, opt["fft_variant"])

    # phase breakdown of one more (untimed) step on the first timed k batch
    phases = None
    if not args.no_trace:
        plan.trace(True)
        plan.solve_bands(kbatch(args.warmup), p.n_bands, allow_nonconv=True)
        tr = plan.trace(False)
        phases = {k: round(v["ms"], 3) for k, v in tr.items()}

    # config 3 as written: the whole path in one bloch_solve_bands call (warm plan)
    path = None
    if not args.no_path and ws == 1:
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e0.record(stream)
        om_path, st_path, status_path = plan.solve_bands(p.k_list, p.n_bands, allow_nonconv=True)
        e1.record(stream)
        torch.cuda.synchronize()
        tp = e0.elapsed_time(e1) / 1000.0
        path = {"n_k": int(nk), "value": nk * p.n_bands / tp, "ms": tp * 1000.0, "status": int(status_path),
                "k_unconverged": int(st_path["k_unconverged"]),
                "k_applies_per_eigenpair": st_path["k_applies"] / (nk * p.n_bands)}

    # the plain FP64 form (the paper's method: shift-invert Lanczos, PCG 1e-10,
    # cuFFT operator) on a near-Gamma and a mid-path batch, the chosen form on
    # the same batches, and the largest frequency difference between the two
    plain = None
    if not args.no_plain and ws == 1 and args.form == "chosen":
        batches = [[1, 2, 3, 4], [20, 21, 22, 23]]
        popt = dict(precision=bloch.FP64, method=bloch.LANCZOS, tol_lin=1e-10, tol_eig=1e-10, max_cg=2000,
                    max_outer=args.max_outer, fft_variant=2, cuda_graph=1)
        pplan = bloch.Plan.from_problem(p, **popt)
        tp = tc = 0.0
        diff = 0.0
        statuses = []
        for bt in batches:
            kb = p.k_list[bt]
            for which, pl_ in (("plain", pplan), ("chosen", plan)):
                e0 = torch.cuda.Event(enable_timing=True)
                e1 = torch.cuda.Event(enable_timing=True)
                torch.cuda.synchronize()
                e0.record(stream)
                om, _, stt = pl_.solve_bands(kb, p.n_bands, allow_nonconv=True)
                e1.record(stream)
                torch.cuda.synchronize()
                dt = e0.elapsed_time(e1) / 1000.0
                statuses.append(int(stt))
                if which == "plain":
                    tp += dt
                    om_plain = om
                else:
                    tc += dt
                    diff = max(diff, float(np.max(np.abs(om / om_plain - 1.0))))
        pplan.close()
        npairs = sum(len(b) for b in batches) * p.n_bands
        plain = {"form": "FP64, shift-invert Lanczos, PCG 1e-10, cuFFT operator (fft_variant 2)",
                 "k_indices": batches, "value": npairs / tp, "chosen_same_batches": npairs / tc,
                 "chosen_over_plain": tp / tc, "max_rel_freq_diff": diff, "statuses": statuses,
                 "unit": "eigenpairs/s"}

    # end to end through the public API with host buffers: plan upload from
    # host arrays, then the same k batches as the timed region (host k lists
    # in, host frequencies out)
    e2e = None
    if not args.no_e2e:
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        plan2 = bloch.Plan.from_problem(p, **opt)
        if lp is not None:
            bloch.set_preconditioner(plan2, lp)
        d2h = 0
        for s in range(args.steps):
            om, _, _ = plan2.solve_bands(kbatch(args.warmup + s), p.n_bands, allow_nonconv=True)
            d2h += om.nbytes
        torch.cuda.synchronize()
        te = time.perf_counter() - t0
        te = max_over_ranks(ws, te)
        plan2.close()
        h2d = p.grain_ids.nbytes + p.C_per_grain.nbytes + p.rho.nbytes + args.steps * kps * 3 * 8
        e2e = {"value": pairs / te, "unit": "eigenpairs/s", "h2d_bytes_per_step": int(h2d // args.steps),
               "d2h_bytes_per_step": int(d2h // args.steps),
               "note": "plan creation from host arrays once, then the timed region's k batches"}

    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu:
        ob = oracle_band_baseline()
        same = gpu_band_same_config(ob["workload"], ob["omega"])
        ta, threads = oracle_sample(p, 1)
        a_per_pair = kap / (args.steps * kps * p.n_bands)
        cpu = {"value": ob["all_cores"]["value"], "unit": "eigenpairs/s", "cores": ob["all_cores"]["cores"],
               "kind": "oracle",
               "sample": (f"measured, not extrapolated: the FP64 oracle's whole band solve of {ob['workload']} "
                          f"({ob['n_k']} k x {ob['n_bands']} bands, grid {ob['grid']}, tol {ob['tol']}), one wave "
                          f"vector per spawned process on {ob['all_cores']['processes']} processes, "
                          f"{ob['all_cores']['wall_s']:.1f} s wall; that config differs from the GPU's 128^3 "
                          f"workload (see same_config_gpu for ours on it)"),
               "one_core": ob["one_core"], "same_config_gpu": same,
               "workload_128_estimate": {
                   "value": 1.0 / (ta * a_per_pair), "s_per_apply": ta,
                   "note": "estimate, not a measurement: oracle seconds per A_k apply at 128^3 times the "
                           "K-applies per eigenpair of the timed GPU form"}}

    if rank == 0:
        valid = k_unconv == 0 and all(st == 0 for st in status_all)
        line = {"metric": metric_of(p.grid), "value": value, "unit": "eigenpairs/s", "n_gpus": ws, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": 1000.0 * t / args.steps, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": "f32" if prec == bloch.FP32 else "f64",
                "data": "synthetic", "valid": valid,
                "config": {"workload": args.workload, "grid": list(p.grid), "grains": int(p.G),
                           "n_bands": p.n_bands, "n_k_path": int(nk), "k_per_step": kps,
                           "k_covered": len(covered),
                           "form": args.form, "tol_eig": opt["tol_eig"], "tol_lin": opt["tol_lin"],
                           "fft_variant": opt["fft_variant"], "cuda_graph": opt["cuda_graph"],
                           "tensor_gram": opt.get("tensor_gram", 0), "block": opt.get("block", 0),
                           "ncv": opt.get("ncv", 0), "k_batch": opt.get("k_batch", 0), "hybrid_tol": opt.get("hybrid_tol", 0.0),
                           "refine_arith": opt.get("refine_arith", 0),
                           "method": {0: "lanczos", 1: "subspace", 2: "lobpcg"}[opt["method"]],
                           "l2": "inputs larger than L2 (one 3-component FP32 vector is %.0f MB)"
                                 % (3 * plan.V * 8 / 1e6)},
                "gpu_launches": int(launches), "clocks": clk, "roofline": roof, "e2e": e2e, "cpu_baseline": cpu,
                "solve_status": {"per_step": status_all, "k_unconverged": k_unconv},
                "solver": {"cg_iterations": cg, "k_applies": kap,
                           "outer_iterations": sum(s["outer_iterations"] for s in stats_all),
                           "max_rel_residual": max(s["max_rel_residual"] for s in stats_all),
                           "k_applies_per_eigenpair": kap / (args.steps * kps * p.n_bands)},
                "path_one_call": path, "plain_baseline": plain,
                "phases_ms": phases, "precond": lp_info}
        print(json.dumps(line), flush=True)
    plan.close()


def main():
    args = parse()
    ws, rank, local = dist_init(args)
    if args.impl == "reference":
        run_reference(args, ws, rank)
    else:
        run_ours(args, ws, rank, local)
    if ws > 1:
        import torch.distributed as dist
        dist.destroy_process_group()


if __name__ == "__main__":
    main()
