#!/usr/bin/env python3
"""Benchmark of the non-local eikonal phase retrieval solve on GB300.

Workload (one step = one full solve from the flat field):
  one monochromatic 2048 x 2048 float32 projection of 200 seeded ellipsoids
  (bone / soft tissue / voids), E = 80 keV, L = 30 m, p = 20 um (1-8 px ray
  shifts), 1e4 photons/px Poisson noise, 50 non-local iterations, omega 0.4.

Prints ONE JSON line (rank 0): value = 2048^2-equivalent projections solved
per second over all ranks, with the kernel roofline, the end-to-end figure
through the C ABI with host buffers, the batched-vs-plain factor, SM clocks
sampled during the timed region, and the FP64 oracle timed on host cores.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

With --gpus N > 1 (under torchrun) every rank solves its own projection
(independent units, no collective on the data path) and the slowest rank's
time sets the figure.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "2048² projections/s to fixed residual, % HBM roofline, batched vs plain GPU"
UNIT = "projections/s"
WORKLOAD = ("ellipsoids_mono_2048: 1 projection 2048x2048 f32, 200 ellipsoids (bone/tissue/void), "
            "E=80 keV, L=30 m, p=20 um, 1e4 photons/px, 50 non-local iterations, omega=0.4")
REF_PIX = 2048 * 2048
PHANTOM_SEED, NOISE_SEED = 2000, 7   # the headline projection of rank 0


def bench_config(wl, world: int) -> dict:
    """The workload description, identical in both arms."""
    return {"workload": WORKLOAD, "nx": wl.nx, "ny": wl.ny, "n_lines": 1,
            "n_iter": wl.n_iter, "omega": wl.omega,
            "seeds": {"phantom": PHANTOM_SEED, "noise": NOISE_SEED, "per_rank": "+ rank"},
            "l2": "flushed between steps (256 MiB write, untimed); working set of one "
                  "projection (~64 MiB) stays L2-resident within a solve",
            "parallelism": f"replicas x{world}"}


# --------------------------------------------------------------------------
# helpers
# --------------------------------------------------------------------------

def _args():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=200)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-iters", type=int, default=4,
                    help="oracle iterations in the CPU-baseline sample")
    ap.add_argument("--ncu-case", action="store_true",
                    help="profiling case for ncu: --batch projections of the workload, "
                         "--warmup + --steps solves of --iters iterations, no report")
    ap.add_argument("--batch", type=int, default=4)
    ap.add_argument("--iters", type=int, default=2)
    ap.add_argument("--lines", type=int, default=1,
                    help="ncu case: 1 = the monochromatic workload, 8 = the polychromatic one")
    ap.add_argument("--oversample", type=int, default=1,
                    help="ncu case: solve on a grid oversampled by this factor (non-local)")
    ap.add_argument("--tuning", default="",
                    help="ncu case: kernel choices as printed by a --tuned run (JSON), applied "
                         "instead of tuning under the profiler")
    ap.add_argument("--tuned", action="store_true",
                    help="ncu case: an autotuned plan (tuned by the first warm-up solve); the "
                         "steps run inside the NVTX range 'steps' (ncu --nvtx --nvtx-include "
                         "steps/)")
    return ap.parse_args()


def _dist():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


def rank_seed(rank: int) -> int:
    """Replica sharding: every rank solves its own projection (independent
    units, no data exchanged between ranks)."""
    return PHANTOM_SEED + rank


def max_over_ranks(x: float, world: int, device=None) -> float:
    """The slowest rank's figure (the job is done when every rank is)."""
    if world <= 1:
        return float(x)
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def whole_job_rate(ms_per_step: float, world: int, npix: int) -> float:
    """2048^2-equivalent projections per second over all ranks: each of the
    `world` ranks solves one npix projection per step."""
    return world * (npix / REF_PIX) / (ms_per_step / 1000.0)


def _peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            pk = json.load(f)
        return float(pk["hbm_gbs"]), "measured"
    except Exception:
        return 6800.0, "fallback"


class ClockSampler:
    """nvidia-smi clock / throttle sampling at 200 ms during a region."""

    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, local_rank: int):
        vis = os.environ.get("CUDA_VISIBLE_DEVICES", "")
        ids = [v.strip() for v in vis.split(",") if v.strip()]
        self.idx = ids[local_rank] if local_rank < len(ids) else str(local_rank)
        self.proc = None
        self.t0 = self.t1 = 0.0

    def start(self):
        try:
            self.proc = subprocess.Popen(
                ["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                 "-lms", "200", "-i", str(self.idx)],
                stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
        except Exception:
            self.proc = None
        self.t0 = time.time()

    def stop(self):
        self.t1 = time.time()
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"],
                    "samples": 0}
        self.proc.terminate()
        try:
            out, _ = self.proc.communicate(timeout=5)
        except Exception:
            self.proc.kill()
            out = ""
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in out.splitlines():
            parts = [x.strip() for x in line.split(",")]
            if len(parts) < 9:
                continue
            try:
                sm.append(float(parts[1]))
                mx.append(float(parts[2]))
            except ValueError:
                continue
            for nm, v in zip(names, parts[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def _traffic(kernel: str, table: str = "dram_traffic.txt"):
    """Per-launch figure of `kernel` from a committed ncu table (DRAM bytes,
    or warp instructions), or None when the library sources changed since
    that capture."""
    path = os.path.join(ROOT, "profiles", table)
    if not os.path.exists(path):
        return None
    from paper_2601_22793_gb300 import build as B
    dig = B._digest()
    with open(path) as f:
        for line in f:
            parts = line.split()
            if len(parts) >= 4 and not line.startswith("#") and parts[0] == kernel:
                if parts[3] != dig[:16]:
                    return None
                return float(parts[2])
    return None


# --------------------------------------------------------------------------
# algorithmic bytes per pixel per launch (float32 maps, one projection)
# --------------------------------------------------------------------------

def kernel_bytes_per_px(ns: int) -> dict:
    """Unavoidable reads + writes of each kernel of one iteration.
    mono (float): splat reads T and D and writes the residual D - P;
                  row_fwd reads T and the residual, writes the packed half
                  spectrum (4 B/px); col reads + writes the spectrum;
                  row_inv reads the spectrum and T, writes T'.
    n_s lines:    splat reads T and D, writes D - P and the split residuals
                  r_s (and P, which only the passes over the long-shift
                  sources read: not counted); row_fwd reads T and r_s, writes
                  n_s spectra; col 8 B/px/line; row_inv reads n_s spectra and
                  T, writes T'."""
    if ns == 1:
        return {"splat": 12, "row_fwd": 12, "col": 8, "row_inv": 12}
    return {"splat": 12 + 4 * ns, "row_fwd": 4 + 8 * ns, "col": 8 * ns, "row_inv": 8 + 4 * ns}


def model_bytes_per_px(ns: int) -> int:
    """The per-iteration streaming model of the hot path, one pass per step:
    splat (read T, write P [and P_s]), gather (read T, D, P [, P_s], write g_s),
    R2C rows, columns, C2R rows with the update: 52 B/px for one line,
    28 + 32 n_s for n_s lines.  The fused kernels move fewer bytes (44 for one
    line; kernel_bytes_per_px); fractions on both are reported."""
    return 52 if ns == 1 else 28 + 32 * ns


def convergence(info) -> dict:
    """Residual and relative update of the headline solve, and the first
    iteration at which the relative update kappa falls to each level."""
    kh = np.asarray(info["kappa_hist"][0])
    reach = {}
    for lev in (1e-2, 5e-3, 2e-3, 1e-3):
        hit = np.nonzero(kh[:int(info["iters"][0])] <= lev)[0]
        reach[f"{lev:g}"] = int(hit[0]) + 1 if hit.size else None
    return {"rho_final": round(float(info["rho"][0]), 6), "kappa_final": float(info["kappa"][0]),
            "iterations_to_kappa": reach}


def _events_ms(fn, torch, reps=1, warm=1):
    """Median CUDA-event time of fn on the current stream (after warm calls)."""
    stream = torch.cuda.current_stream()
    for _ in range(warm):
        fn()
    torch.cuda.synchronize()
    ts = []
    for _ in range(reps):
        a = torch.cuda.Event(enable_timing=True)
        b = torch.cuda.Event(enable_timing=True)
        a.record(stream)
        fn()
        b.record(stream)
        b.synchronize()
        ts.append(a.elapsed_time(b))
    return float(np.median(ts))


def uneven_batch(epr, ph, torch, peak, n_proj=512, max_iter=80, deterministic=False, tol=2e-3):
    """Batched solve of projections of uneven sizes in one call: sizes drawn
    uniformly from {1024x1024, 2048x1536, 2048x2048, 3072x2048} (nx x ny), 4
    lines 60-160 keV, each projection's thickness scaled so that its largest
    shift is U[0.2, 10] px, each solved until kappa <= tol or max_iter.  Under
    Poisson(1e4) noise kappa levels off near 1e-3 (the oracle: 250 iterations
    of such projections), so the tolerance is 2e-3, where projections retire
    between about 40 and 80 iterations; a tolerance of 1e-4 would retire
    none.  Data: 8 seeded 60-ellipsoid phantoms per size, the library's
    forward model and Poisson(1e4) noise drawn on the device (seeded)."""
    sizes = [(1024, 1024), (2048, 1536), (2048, 2048), (3072, 2048)]
    E4, d4, b4, w4 = ph.spectrum(4, 60.0, 160.0, 95.0, 30.0, ph.BONE[0], ph.BONE[1], 80.0, 4000)
    pixel, L, photons, n_base = 20e-6, 30.0, 1e4, 8
    cmax = L * float(np.max(d4)) / pixel ** 2       # shift per thickness step, largest line
    base = []
    for si, (nx, ny) in enumerate(sizes):
        row = []
        for k in range(n_base):
            ells = ph.random_ellipsoids(ny, nx, 60, 8.0, 120.0, seed=4200 + 10 * si + k)
            t = ph.project_ellipsoids(ells, ny, nx, pixel)
            gy, gx = np.gradient(t)
            row.append((torch.from_numpy(t.astype(np.float32)).cuda(),
                        cmax * max(np.abs(gx).max(), np.abs(gy).max())))
        base.append(row)
    g = ph.rng(4100)
    gen = torch.Generator(device="cuda").manual_seed(4101)
    Ds, Ts, shapes, targets = [], [], [], []
    plans = [epr.Plan(nx, ny, pixel, L, E4, d4, b4, w4, max_shift_px=6, overflow_capacity=1 << 18)
             for nx, ny in sizes]
    for j in range(n_proj):
        si, k = int(g.integers(4)), int(g.integers(n_base))
        target = float(g.uniform(0.2, 10.0))
        t, umax = base[si][k]
        tj = t * (target / umax)
        P = torch.empty_like(tj)
        epr.epr_forward(plans[si].handle, tj, P)
        Ds.append(torch.poisson(photons * P.clamp_min(0), generator=gen) / photons)
        Ts.append(torch.empty_like(tj))
        shapes.append(sizes[si])
        targets.append(target)
    for q in plans:
        q.close()
    bh = epr.epr_batch_create(pixel, L, E4, d4, b4, w4, max_shift_px=6, autotune=True,
                              overflow_capacity=1 << 18, deterministic=deterministic)
    info = {}

    def call():
        info.update(epr.epr_solve_nonlocal_batched(bh, Ds, Ts, n_iter=max_iter, omega=0.4,
                                                   tol=tol))

    ms = _events_ms(call, torch, reps=1, warm=1)   # the warm call also tunes the splat
    epr.epr_batch_destroy(bh)
    iters = np.asarray(info["iters"], int)
    npx = np.asarray([nx * ny for nx, ny in shapes], float)
    bpp = model_bytes_per_px(4)
    gbs = float((iters * npx).sum()) * bpp / (ms * 1e-3) / 1e9
    hist = np.bincount(np.minimum(iters // 10, max_iter // 10), minlength=max_iter // 10 + 1)
    conv = iters < max_iter
    return {"projections": n_proj, "sizes_nx_ny": sizes, "n_lines": 4, "tol_kappa": tol,
            "max_iter": max_iter, "max_shift_px": "U[0.2, 10] per projection",
            "deterministic": bool(deterministic), "ms_per_call": round(ms, 1),
            "equiv_2048sq_projections_per_s": round(float(npx.sum()) / REF_PIX / (ms * 1e-3), 3),
            "retired_by_kappa": int(conv.sum()),
            "iterations_histogram_per_10": hist.tolist(),
            "mean_iterations": round(float(iters.mean()), 2),
            "hbm": {"alg_bytes_per_px_per_iter": bpp, "achieved_gbs": round(gbs, 1), "peak": peak,
                    "frac": round(gbs / peak, 4),
                    "note": "algorithmic bytes of the iterations each projection ran / time"},
            "kappa_of_unconverged_max": float(np.max(np.asarray(info["kappa"])[~conv]))
            if (~conv).any() else None}


def unrolled_vjp(epr, ph, torch, peak, batch=16, n_iter=30):
    """Reverse mode through n_iter unrolled 8-line non-local iterations of a
    batch of 2048^2 projections (the rotated ellipsoid phantom at `batch`
    angles), with and without checkpointing of the iterates."""
    wp, ells, angles = ph.ellipsoids_poly()
    taus = [ph.project_ellipsoids(ells, wp.ny, wp.nx, wp.pixel, angles[4 * j % len(angles)])
            for j in range(batch)]
    plan = epr.Plan(wp.nx, wp.ny, wp.pixel, wp.L, wp.energy_keV, wp.delta, wp.beta, wp.weights)
    T = torch.from_numpy(np.stack(taus).astype(np.float32)).cuda()
    P = torch.empty_like(T)
    epr.epr_forward(plan.handle, T, P, batch=batch)
    gen = torch.Generator(device="cuda").manual_seed(5001)
    D = torch.poisson(wp.photons * P.clamp_min(0), generator=gen) / wp.photons
    Tbar = torch.randn(T.shape, device="cuda", generator=gen)
    t0b, Db = torch.empty_like(T), torch.empty_like(T)
    ns = int(np.size(wp.energy_keV))
    out = {"workload": f"{batch} x 2048x2048, 8 lines, {n_iter} unrolled iterations from the flat "
                       "field, omega 0.4; gradients in T0, D, L, delta_s, beta_s",
           "batch": batch, "n_iter": n_iter}
    for ck in (0, 5):
        ms = _events_ms(lambda: epr.epr_solve_vjp(plan.handle, D, Tbar, ns, n_iter, omega=wp.omega,
                                                  checkpoint_every=ck, batch=batch, T0_bar=t0b,
                                                  D_bar=Db, scalars=True), torch, reps=1, warm=1)
        out["ms_all_iterates_kept" if ck == 0 else "ms_checkpoint_every_5"] = round(ms, 1)
    fwd = _events_ms(lambda: epr.epr_solve_nonlocal(plan.handle, D, T, batch=batch, n_iter=n_iter,
                                                    omega=wp.omega, want_info=False), torch, reps=1)
    out["ms_forward_solve_only"] = round(fwd, 1)
    out["projections_per_s"] = round(batch / (out["ms_all_iterates_kept"] * 1e-3), 3)
    plan.close()
    return out


def xspec_solve(epr, ph, torch, timeit):
    """One 2048^2 8-line projection solved with an x-dependent spectrum (a
    five-knot table across the columns: weights +-30 %, delta and beta +-20 %),
    50 iterations, against the same solve with the uniform spectrum."""
    wp, ells, angles = ph.ellipsoids_poly()
    tau = ph.project_ellipsoids(ells, wp.ny, wp.nx, wp.pixel, angles[8])
    ns = int(np.size(wp.energy_keV))
    g = ph.rng(6001)
    X = np.linspace(0.0, wp.nx - 1.0, 5)
    W = wp.weights[:, None] * g.uniform(0.7, 1.3, size=(ns, 5))
    Dl = wp.delta[:, None] * g.uniform(0.8, 1.2, size=(ns, 5))
    Bt = wp.beta[:, None] * g.uniform(0.8, 1.2, size=(ns, 5))
    plan = epr.Plan(wp.nx, wp.ny, wp.pixel, wp.L, wp.energy_keV, wp.delta, wp.beta, wp.weights)
    T = torch.from_numpy(tau.astype(np.float32)).cuda()
    P = torch.empty_like(T)
    epr.epr_plan_set_xspec(plan.handle, X, W, Dl, Bt)
    epr.epr_forward(plan.handle, T, P)
    gen = torch.Generator(device="cuda").manual_seed(6002)
    D = torch.poisson(wp.photons * P.clamp_min(0), generator=gen) / wp.photons
    ms_x = timeit(lambda: epr.epr_solve_nonlocal(plan.handle, D, T, n_iter=wp.n_iter,
                                                 omega=wp.omega, want_info=False), reps=3)
    epr.epr_plan_set_xspec(plan.handle)
    ms_u = timeit(lambda: epr.epr_solve_nonlocal(plan.handle, D, T, n_iter=wp.n_iter,
                                                 omega=wp.omega, want_info=False), reps=3)
    plan.close()
    return {"workload": "ellipsoids_poly_2048, 1 projection, 8 lines, 50 iterations, 5-knot "
                        "x-dependent table", "ms_per_solve": round(ms_x, 3),
            "ms_per_solve_uniform_spectrum": round(ms_u, 3),
            "note": "the x-dependent path runs the kernels with per-column constants"}


# --------------------------------------------------------------------------
# our arm
# --------------------------------------------------------------------------

def run_ours(a):
    import torch

    from paper_2601_22793_gb300 import build as B
    from paper_2601_22793_gb300 import epr
    from paper_2601_22793_gb300 import phantoms as ph

    rank, world, local = _dist()
    if a.ncu_case:
        torch.cuda.set_device(local)
        return ncu_case(a)
    # The CPU-baseline leg runs first, before any CUDA work of this process:
    # it times the oracle on the host cores and, while doing so, makes the
    # seeded data D of the headline projection with the oracle's forward model
    # (the same D the reference arm solves).  Without that leg (N > 1, or
    # --no-cpu-baseline) every rank makes its data with the library's forward.
    cpu, D_oracle = None, None
    if rank == 0 and world == 1 and not a.no_cpu_baseline:
        cpu, D_oracle = cpu_baseline(a.cpu_iters)
    torch.cuda.set_device(local)
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("nccl", device_id=torch.device("cuda", local))
    B.build()
    epr.load()

    wl, tau = ph.ellipsoids_mono(seed=rank_seed(rank))
    npix = wl.nx * wl.ny
    # the autotuner picks the splat tile and reach, the column plan and tile width and
    # the row passes' blocks per SM during the first (warm-up) solve
    plan = epr.Plan(wl.nx, wl.ny, wl.pixel, wl.L, wl.energy_keV, wl.delta, wl.beta, wl.weights,
                    autotune=True)
    stream = torch.cuda.current_stream()
    Tt = torch.from_numpy(tau.astype(np.float32)).cuda()
    Pt = torch.empty_like(Tt)
    if D_oracle is not None:
        D_host = D_oracle
        data_src = ("synthetic: seeded ellipsoid phantom, D = FP64 oracle forward + Poisson(1e4) "
                    "(made by the CPU-baseline leg; the reference arm solves the same D)")
    else:
        # the library's own forward model on the device, counting noise on the host
        epr.epr_forward(plan.handle, Tt, Pt)
        D_host = ph.poisson(Pt.cpu().numpy(), wl.photons, NOISE_SEED + rank).astype(np.float32)
        data_src = "synthetic: seeded ellipsoid phantom, D = library forward + Poisson(1e4)"
    D = torch.from_numpy(D_host).cuda()
    T = torch.empty_like(D)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device="cuda")

    def solve():
        epr.epr_solve_nonlocal(plan.handle, D, T, n_iter=wl.n_iter, omega=wl.omega,
                               want_info=False)

    for _ in range(a.warmup):
        flush.zero_()
        solve()
    torch.cuda.synchronize()

    def barrier():
        if world > 1:
            torch.distributed.barrier()

    clocks = ClockSampler(local)
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(a.steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(a.steps)]
    barrier()
    torch.cuda.synchronize()
    clocks.start()
    l0 = epr.epr_launch_count()
    for k in range(a.steps):
        flush.zero_()                     # L2 flush between steps (untimed)
        starts[k].record(stream)
        solve()
        ends[k].record(stream)
    torch.cuda.synchronize()
    launches = epr.epr_launch_count() - l0
    # keep sampling clocks for at least ~1.5 s of the same loop when the
    # timed region itself was shorter than a few nvidia-smi periods
    t_region = time.time() - clocks.t0
    extra = 0
    while time.time() - clocks.t0 < 1.5:
        flush.zero_()
        solve()
        extra += 1
    torch.cuda.synchronize()
    clk = clocks.stop()
    barrier()
    step_ms = [s.elapsed_time(e) for s, e in zip(starts, ends)]
    ms = max_over_ranks(float(np.mean(step_ms)), world, device="cuda")
    value = whole_job_rate(ms, world, npix)

    # convergence figures of this workload
    info = epr.epr_solve_nonlocal(plan.handle, D, T, n_iter=wl.n_iter, omega=wl.omega)
    tuning = epr.epr_plan_get_tuning(plan.handle)

    # kernel roofline: the same solves with per-kernel CUDA events
    epr.epr_profile_enable(plan.handle, True)
    n_prof = max(3, min(8, a.steps))
    for _ in range(n_prof):
        flush.zero_()
        solve()
    torch.cuda.synchronize()
    prof = epr.epr_profile_read(plan.handle)
    epr.epr_profile_enable(plan.handle, False)
    bpp = kernel_bytes_per_px(1)
    peak, peak_src = _peaks()
    per_kernel = {}
    for kname, (cnt, tot) in prof.items():
        if cnt == 0 or kname not in bpp:
            continue
        avg_ms = tot / cnt
        alg = bpp[kname] * npix
        per_kernel[kname] = {"launches": cnt, "avg_us": round(avg_ms * 1e3, 3),
                             "alg_bytes": alg, "gbs": round(alg / (avg_ms * 1e-3) / 1e9, 1),
                             "share": 0.0}
    tot_ms = sum(v["avg_us"] * v["launches"] for v in per_kernel.values())
    for v in per_kernel.values():
        v["share"] = round(v["avg_us"] * v["launches"] / tot_ms, 4) if tot_ms else 0.0
    dom = max(per_kernel, key=lambda k: per_kernel[k]["avg_us"] * per_kernel[k]["launches"])
    dk = per_kernel[dom]
    iter_bytes = sum(bpp.values()) * npix
    iter_us = sum(v["avg_us"] for v in per_kernel.values())
    tr = _traffic(dom)
    live_us = ms * 1e3 / wl.n_iter   # one iteration of the timed (graph-replayed) solve
    model_bytes = model_bytes_per_px(1) * npix
    roofline = {"bound": "hbm", "kernel": dom, "achieved": dk["gbs"], "peak": peak,
                "unit": "GB/s", "frac": round(dk["gbs"] / peak, 4),
                "traffic": tr, "peak_source": f"{peak_src} hbm_gbs",
                "alg_bytes_per_launch": dk["alg_bytes"],
                "timing": "per-kernel CUDA events recorded inside a profiled graph of the same "
                          "solve; the event records serialise the launches (no programmatic "
                          "overlap), so per-kernel figures are serialised ones",
                "iteration_serialised": {"alg_bytes": iter_bytes, "kernel_us": round(iter_us, 2),
                                         "gbs": round(iter_bytes / (iter_us * 1e-6) / 1e9, 1),
                                         "frac": round(iter_bytes / (iter_us * 1e-6) / 1e9 / peak, 4)},
                "iteration_live": {"alg_bytes": model_bytes, "us": round(live_us, 2),
                                   "gbs": round(model_bytes / (live_us * 1e-6) / 1e9, 1),
                                   "frac": round(model_bytes / (live_us * 1e-6) / 1e9 / peak, 4),
                                   "frac_fused_kernel_bytes":
                                       round(iter_bytes / (live_us * 1e-6) / 1e9 / peak, 4),
                                   "note": "ms_per_step / n_iter of the timed solves; bytes of "
                                           "the 52 B/px model (fused kernels: 44 B/px)"},
                "kernels": per_kernel}
    # the bound the kernels actually meet: instruction issue (4 warp instructions
    # per clock per SM), with the instructions ncu counted per launch
    nsm = torch.cuda.get_device_properties(local).multi_processor_count
    issue_peak = nsm * 4 * clk["sm_mhz"] * 1e6 / 1e9 if clk["sm_mhz"] else None
    issue = {}
    for kname, v in per_kernel.items():
        ninst = _traffic(kname, "instructions.txt")
        if ninst is None or not issue_peak:
            issue[kname] = None
            continue
        ach = ninst / (v["avg_us"] * 1e-6) / 1e9
        issue[kname] = {"warp_inst_per_launch": int(ninst), "achieved_ginst_s": round(ach, 1),
                        "frac": round(ach / issue_peak, 4)}
    roofline["issue"] = {"peak_ginst_s": round(issue_peak, 1) if issue_peak else None,
                         "peak_source": f"{nsm} SMs x 4 schedulers x sampled SM clock",
                         "kernels": issue,
                         "note": "informational: the measured bound of these kernels is "
                                 "instruction issue and load latency, not HBM"}

    # end to end through the C ABI with pinned host buffers
    Dh = torch.from_numpy(D_host).pin_memory()
    Th = torch.empty((wl.ny, wl.nx), dtype=torch.float32).pin_memory()
    for _ in range(3):
        epr.epr_solve_nonlocal(plan.handle, Dh, Th, n_iter=wl.n_iter, omega=wl.omega,
                               want_info=False)
    torch.cuda.synchronize()
    n_e2e = max(5, min(50, a.steps))
    e_start = torch.cuda.Event(enable_timing=True)
    e_end = torch.cuda.Event(enable_timing=True)
    e_times = []
    for _ in range(n_e2e):
        flush.zero_()
        e_start.record(stream)
        epr.epr_solve_nonlocal(plan.handle, Dh, Th, n_iter=wl.n_iter, omega=wl.omega,
                               want_info=False)
        e_end.record(stream)
        e_end.synchronize()
        e_times.append(e_start.elapsed_time(e_end))
    e_ms = max_over_ranks(float(np.mean(e_times)), world, device="cuda")
    e2e = {"value": round(whole_job_rate(e_ms, world, npix), 3), "unit": UNIT,
           "h2d_bytes_per_step": int(D_host.nbytes), "d2h_bytes_per_step": int(Th.numel() * 4),
           "ms_per_step": round(e_ms, 4)}

    # batched (one call, 32 projections, graph) vs plain (one projection per call, no
    # graph): 8 phantoms, each under 4 independent counting-noise draws
    nb, n_ph = 32, 8
    Ds = []
    for j in range(n_ph):
        _, tk = ph.ellipsoids_mono(seed=3000 + 100 * rank + j)
        epr.epr_forward(plan.handle, torch.from_numpy(tk.astype(np.float32)).cuda(), Pt)
        Pj = Pt.cpu().numpy()
        for r in range(nb // n_ph):
            Ds.append(ph.poisson(Pj, wl.photons, 50 + j * (nb // n_ph) + r).astype(np.float32))
    Db = torch.from_numpy(np.stack(Ds)).cuda()
    Tb = torch.empty_like(Db)
    plain = epr.Plan(wl.nx, wl.ny, wl.pixel, wl.L, wl.energy_keV, wl.delta, wl.beta, wl.weights,
                     use_graphs=False, autotune=True)
    # the batch has its own plan, tuned on its first (untimed) call
    bplan = epr.Plan(wl.nx, wl.ny, wl.pixel, wl.L, wl.energy_keV, wl.delta, wl.beta, wl.weights,
                     autotune=True)

    def batched():
        epr.epr_solve_nonlocal(bplan.handle, Db, Tb, batch=nb, n_iter=wl.n_iter, omega=wl.omega,
                               want_info=False)

    def plain_run():
        for k in range(nb):
            epr.epr_solve_nonlocal(plain.handle, Db[k], Tb[k], n_iter=wl.n_iter,
                                   omega=wl.omega, want_info=False)

    def timeit(fn, reps=5):
        fn()
        torch.cuda.synchronize()
        ts = []
        for _ in range(reps):
            flush.zero_()
            s0 = torch.cuda.Event(enable_timing=True)
            s1 = torch.cuda.Event(enable_timing=True)
            s0.record(stream)
            fn()
            s1.record(stream)
            s1.synchronize()
            ts.append(s0.elapsed_time(s1))
        return float(np.median(ts))

    t_b = timeit(batched)
    t_p = timeit(plain_run)
    btuning = epr.epr_plan_get_tuning(bplan.handle)
    plain.close()
    bplan.close()
    it_bytes = model_bytes_per_px(1) * npix   # algorithmic bytes per iteration (model)
    b_gbs = it_bytes * wl.n_iter * nb / (t_b * 1e-3) / 1e9
    f_gbs = sum(kernel_bytes_per_px(1).values()) * npix * wl.n_iter * nb / (t_b * 1e-3) / 1e9
    bvp = {"batch": nb, "batched_ms": round(t_b, 3), "plain_ms": round(t_p, 3),
           "factor": round(t_p / t_b, 3),
           "batched_projections_per_s": round(nb / (t_b * 1e-3), 3),
           "batched_hbm": {"achieved_gbs": round(b_gbs, 1), "peak": peak,
                           "frac": round(b_gbs / peak, 4),
                           "alg_bytes_per_px_per_iter": model_bytes_per_px(1),
                           "frac_fused_kernel_bytes": round(f_gbs / peak, 4),
                           "note": "algorithmic bytes of all kernels of all iterations / time; "
                                   f"{nb} x 64 MiB working set exceeds L2"},
           "tuning": btuning,
           "plain": "one projection per call, kernels launched one by one (no graph)",
           "batched": "one call for all projections, iteration loop replayed as a CUDA graph"}

    # the same workload with the local O(L^2) closure, and an 8-line polychromatic solve
    local_ms = timeit(lambda: epr.epr_solve_local(plan.handle, D, T, order=2, n_iter=wl.n_iter,
                                                  omega=wl.omega, want_info=False))
    other = {"local_closure_order2": {"ms_per_solve": round(local_ms, 3),
                                      "projections_per_s": round(1e3 / local_ms, 3),
                                      "n_iter": wl.n_iter}}
    wp, ells, angles = ph.ellipsoids_poly()
    tp = ph.project_ellipsoids(ells, wp.ny, wp.nx, wp.pixel, angles[rank % len(angles)])
    # tuned like the headline plan: the first solve runs the autotuner, the
    # second captures the graph of the tuned kernels
    pplan = epr.Plan(wp.nx, wp.ny, wp.pixel, wp.L, wp.energy_keV, wp.delta, wp.beta, wp.weights,
                     autotune=True)
    Tp = torch.from_numpy(tp.astype(np.float32)).cuda()
    Pp = torch.empty_like(Tp)
    epr.epr_forward(pplan.handle, Tp, Pp)
    Dp = torch.from_numpy(ph.poisson(Pp.cpu().numpy(), wp.photons, 9).astype(np.float32)).cuda()
    for _ in range(2):
        epr.epr_solve_nonlocal(pplan.handle, Dp, Tp, n_iter=wp.n_iter, omega=wp.omega, want_info=False)
    ptuning = epr.epr_plan_get_tuning(pplan.handle)
    poly_ms = timeit(lambda: epr.epr_solve_nonlocal(pplan.handle, Dp, Tp, n_iter=wp.n_iter,
                                                    omega=wp.omega, want_info=False), reps=3)
    # per-kernel times of the 8-line solve (events in a profiled graph: serialised)
    epr.epr_profile_enable(pplan.handle, True)
    epr.epr_solve_nonlocal(pplan.handle, Dp, Tp, n_iter=wp.n_iter, omega=wp.omega, want_info=False)
    torch.cuda.synchronize()
    pk = epr.epr_profile_read(pplan.handle)
    epr.epr_profile_enable(pplan.handle, False)
    poly_kernels = {k: round(tot * 1e3 / wp.n_iter, 2) for k, (cnt, tot) in pk.items() if cnt}
    # vector-Jacobian product of the 8-line forward (the calibration backward)
    gbar = torch.randn(wp.ny, wp.nx, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    Tbar = torch.empty_like(Tp)
    nlp = int(np.size(wp.energy_keV))
    fwd_ms = timeit(lambda: epr.epr_forward(pplan.handle, Tp, Pp))
    vjp_ms = timeit(lambda: epr.epr_vjp(pplan.handle, Tp, gbar, Tbar, nlp, scalars=False))
    pplan.close()
    other["vjp_polychromatic"] = {"workload": "ellipsoids_poly_2048 forward + VJP, 8 lines, 1 map",
                                  "forward_ms": round(fwd_ms, 3), "vjp_ms": round(vjp_ms, 3)}
    # oversampled internal grids (the paper's operating mode: o = 2 local, 4 non-local):
    # a 2048^2 detector at o = 4 (8192^2 internal) and at o = 2, a 1024^2 one at o = 4
    ovs = {}
    for name, nd, os_, model in (("nonlocal_o4_2048", 2048, 4, 0), ("nonlocal_o2_2048", 2048, 2, 0),
                                 ("nonlocal_o4_1024", 1024, 4, 0), ("local2_o2_2048", 2048, 2, 2)):
        # the 2048^2 phantom subsampled to the detector, replicated to the fine grid
        tf = np.kron(tau[::2048 // nd, ::2048 // nd], np.ones((os_, os_)))
        with epr.Plan(nd, nd, wl.pixel, wl.L, wl.energy_keV, wl.delta, wl.beta, wl.weights,
                      oversample=os_, max_shift_px=8, autotune=True) as op:
            Tf = torch.from_numpy(tf.astype(np.float32)).cuda()
            Pd = torch.empty((nd, nd), device="cuda")
            epr.epr_forward(op.handle, Tf, Pd, model=model)
            Do = torch.from_numpy(ph.poisson(Pd.cpu().numpy(), wl.photons, 11).astype(np.float32)).cuda()
            if model == 0:
                fn = lambda: epr.epr_solve_nonlocal(op.handle, Do, Tf, n_iter=wl.n_iter,
                                                    omega=wl.omega, want_info=False)
            else:
                fn = lambda: epr.epr_solve_local(op.handle, Do, Tf, order=model, n_iter=wl.n_iter,
                                                 omega=wl.omega, want_info=False)
            fn()   # the first solve runs the autotuner; timeit's warm-up captures the graph
            otun = epr.epr_plan_get_tuning(op.handle)
            ms_o = timeit(fn, reps=3)
        o_gbs = model_bytes_per_px(1) * (nd * os_) ** 2 * wl.n_iter / (ms_o * 1e-3) / 1e9
        ovs[name] = {"detector": nd, "oversample": os_, "internal": nd * os_,
                     "model": "nonlocal" if model == 0 else f"local order {model}",
                     "n_iter": wl.n_iter, "ms_per_solve": round(ms_o, 3),
                     "internal_2048sq_equiv_per_s": round((nd * os_) ** 2 / REF_PIX / (ms_o * 1e-3), 3),
                     "hbm": {"alg_bytes_per_internal_px_per_iter": model_bytes_per_px(1),
                             "achieved_gbs": round(o_gbs, 1), "frac": round(o_gbs / peak, 4)},
                     "tuning": otun}
    other["oversampled"] = ovs

    # uneven batch of 512 projections (4 lines, solved to kappa <= 1e-4), float and
    # fixed point; reverse mode through 30 unrolled 8-line iterations of 16
    # projections; the x-dependent spectrum and the second-order model
    other["batched_uneven_512"] = uneven_batch(epr, ph, torch, peak, n_proj=512, max_iter=80)
    other["batched_uneven_fixed_point"] = uneven_batch(epr, ph, torch, peak, n_proj=64,
                                                       max_iter=80, deterministic=True)
    other["unrolled_solve_vjp"] = unrolled_vjp(epr, ph, torch, peak)
    other["xdependent_spectrum"] = xspec_solve(epr, ph, torch, timeit)
    # the same solves on an untuned plan (the library's default choices)
    with epr.Plan(wl.nx, wl.ny, wl.pixel, wl.L, wl.energy_keV, wl.delta, wl.beta, wl.weights) as up:
        other["untuned_plan"] = {
            "ms_per_solve": round(timeit(lambda: epr.epr_solve_nonlocal(
                up.handle, D, T, n_iter=wl.n_iter, omega=wl.omega, want_info=False)), 3),
            "batched_32_ms": round(timeit(lambda: epr.epr_solve_nonlocal(
                up.handle, Db, Tb, batch=nb, n_iter=wl.n_iter, omega=wl.omega, want_info=False),
                reps=3), 3),
            "ms_per_solve_tuned": round(timeit(solve), 3)}
    other["second_order_nonlocal"] = {
        "workload": "the headline projection, non-local model to second order (WKB1 term)",
        "n_iter": wl.n_iter,
        "ms_per_solve": round(timeit(lambda: epr.epr_solve_nonlocal_wkb1(
            plan.handle, D, T, n_iter=wl.n_iter, omega=wl.omega, want_info=False)), 3)}
    nlp8 = int(np.size(wp.energy_keV))
    p_gbs = model_bytes_per_px(nlp8) * wp.nx * wp.ny * wp.n_iter / (poly_ms * 1e-3) / 1e9
    other["polychromatic"] = {"workload": wp.name.replace("x64x", "x1x"),
                              "n_lines": nlp8, "n_iter": wp.n_iter,
                              "ms_per_solve": round(poly_ms, 3),
                              "projections_per_s": round(1e3 / poly_ms, 3),
                              "hbm": {"alg_bytes_per_px_per_iter": model_bytes_per_px(nlp8),
                                      "achieved_gbs": round(p_gbs, 1), "peak": peak,
                                      "frac": round(p_gbs / peak, 4)},
                              "kernels_serialised_us_per_iteration": poly_kernels,
                              "tuning": ptuning}

    out = {"metric": METRIC, "value": round(value, 3), "unit": UNIT, "n_gpus": world,
           "steps": a.steps, "warmup": a.warmup, "ms_per_step": round(ms, 4),
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
           "data": data_src,
           "config": bench_config(wl, world),
           "convergence": convergence(info),
           "tuning": tuning,
           "roofline": roofline, "e2e": e2e, "batched_vs_plain": bvp, "other_workloads": other,
           "gpu_launches": int(launches),
           "clocks": {"sm_mhz": clk["sm_mhz"], "sm_max_mhz": clk["sm_max_mhz"],
                      "reasons": clk["reasons"], "samples": clk["samples"],
                      "window": f"timed region ({t_region:.2f} s) + {extra} extra solves to 1.5 s"}}
    if cpu is not None:
        out["cpu_baseline"] = cpu
    plan.close()
    if rank == 0:
        print(json.dumps(out), flush=True)
    if world > 1:
        torch.distributed.destroy_process_group()


def ncu_case(a):
    """A small case for ncu captures: a batch of projections of the workload
    (4 x 2048^2 keeps the working set above L2), a few short solves."""
    import torch

    from paper_2601_22793_gb300 import build as B
    from paper_2601_22793_gb300 import epr
    from paper_2601_22793_gb300 import phantoms as ph

    B.build()
    epr.load()
    if a.lines > 1:   # the rotated 8-line phantom at a.batch angles
        wl, ells, angles = ph.ellipsoids_poly(n_lines=a.lines)
        taus = [ph.project_ellipsoids(ells, wl.ny, wl.nx, wl.pixel, angles[k]) for k in range(a.batch)]
    else:
        wl, _ = ph.ellipsoids_mono(seed=2000)
        taus = [ph.ellipsoids_mono(seed=2000 + k)[1] for k in range(a.batch)]
    os_ = max(1, a.oversample)
    n = wl.nx
    if os_ > 1:   # the detector of the workload, an internal grid o times finer
        taus = [np.kron(t, np.ones((os_, os_))) for t in taus]
    plan = epr.Plan(n, n, wl.pixel, wl.L, wl.energy_keV, wl.delta, wl.beta, wl.weights,
                    oversample=os_, max_shift_px=8 if os_ > 1 else 4, autotune=a.tuned)
    Tt = torch.from_numpy(np.stack(taus).astype(np.float32)).cuda()
    P = torch.empty((a.batch, n, n), device="cuda")
    epr.epr_forward(plan.handle, Tt, P, batch=a.batch)
    D = P.clamp_min(0) + 0.01 * torch.randn_like(P)
    T = torch.empty_like(Tt)
    if a.tuning:
        epr.epr_plan_set_tuning(plan.handle, json.loads(a.tuning))
    for k in range(a.warmup + a.steps):
        if k == a.warmup:
            torch.cuda.synchronize()
            torch.cuda.nvtx.range_push("steps")
        epr.epr_solve_nonlocal(plan.handle, D, T, batch=a.batch, n_iter=a.iters,
                               omega=wl.omega, want_info=False)
    torch.cuda.synchronize()
    if a.steps > 0:
        torch.cuda.nvtx.range_pop()
    if a.tuned or a.tuning:
        print("tuning:", json.dumps(epr.epr_plan_get_tuning(plan.handle)))
    plan.close()
    print(f"ncu case done: batch {a.batch}, {a.warmup + a.steps} solves of {a.iters} iterations")


# --------------------------------------------------------------------------
# oracle timings (CPU baseline and the reference arm)
# --------------------------------------------------------------------------

def _oracle_workload():
    """The headline projection as both arms solve it: the seeded phantom, its
    FP64 oracle forward model and Poisson(1e4) counting noise (float32)."""
    from oracle import oracle as O
    from paper_2601_22793_gb300 import phantoms as ph
    O.build()
    wl, tau = ph.ellipsoids_mono(seed=PHANTOM_SEED)
    ln = O.Lines(wl.energy_keV, wl.delta, wl.beta, wl.weights, wl.L, wl.pixel)
    D = ph.poisson(O.forward(ln, tau), wl.photons, NOISE_SEED).astype(np.float32)
    return O, wl, ln, D


def _cpu_model() -> str:
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.split(":")[0].strip() in ("Model name", "Model"):
                name = line.split(":", 1)[1].strip()
                if name and not name.isdigit():
                    return name
    except Exception:
        pass
    import platform
    return platform.processor() or platform.machine()


def _oracle_sample(n_it: int, D) -> float:
    """Seconds of n_it iterations of the oracle's solve of the headline
    workload (one process, one thread)."""
    from oracle import oracle as O
    from paper_2601_22793_gb300 import phantoms as ph
    wl, _ = ph.ellipsoids_mono(seed=PHANTOM_SEED)
    ln = O.Lines(wl.energy_keV, wl.delta, wl.beta, wl.weights, wl.L, wl.pixel)
    t0 = time.perf_counter()
    O.solve(ln, np.asarray(D, np.float64), n_iter=n_it, omega=wl.omega)
    return time.perf_counter() - t0


UNEVEN_SIZES = [(1024, 1024), (2048, 1536), (2048, 2048), (3072, 2048)]   # (nx, ny)


def _oracle_other_configs(band: int = 128) -> dict:
    """Single-threaded oracle timings of the other configurations, on bounded
    samples: the 256^2 sphere solve in full (20 iterations); one iteration of
    the 8-line 2048^2 solve on a band of rows, scaled by pixel count and to 50
    iterations; one iteration of the 4-line solve of each uneven size on a band,
    scaled by pixel count to a 2048^2-equivalent iteration of the uniform size
    mix.  Every iteration of a solve does the same work, so the scaling is
    linear."""
    from oracle import oracle as O
    from paper_2601_22793_gb300 import phantoms as ph
    out = {}
    wl, tau = ph.spheres_mono_256()
    ln = O.Lines(wl.energy_keV, wl.delta, wl.beta, wl.weights, wl.L, wl.pixel)
    D = ph.poisson(O.forward(ln, tau), wl.photons, 3)
    t0 = time.perf_counter()
    O.solve(ln, D, n_iter=wl.n_iter, omega=wl.omega)
    t = time.perf_counter() - t0
    out["spheres_mono_256"] = {"n_iter": wl.n_iter, "s_per_solve": round(t, 4),
                               "projections_per_s": round(1.0 / t, 4), "cores": 1,
                               "sample": "the full solve"}
    wp, ells, angles = ph.ellipsoids_poly()
    y0 = wp.ny // 2 - band // 2
    tp = ph.project_ellipsoids(ells, wp.ny, wp.nx, wp.pixel, angles[0])[y0:y0 + band]
    lp = O.Lines(wp.energy_keV, wp.delta, wp.beta, wp.weights, wp.L, wp.pixel)
    Dp = ph.poisson(O.forward(lp, tp), wp.photons, 9)
    t0 = time.perf_counter()
    O.solve(lp, Dp, n_iter=1, omega=wp.omega)
    it_full = (time.perf_counter() - t0) * wp.ny / band
    out["ellipsoids_poly_2048x8"] = {
        "n_lines": int(np.size(wp.energy_keV)), "s_per_iteration": round(it_full, 3),
        "projections_per_s": round(1.0 / (it_full * wp.n_iter), 6), "cores": 1,
        "sample": f"1 iteration on rows {y0}..{y0 + band - 1} of the 2048x2048 projection, "
                  f"scaled by pixel count and to {wp.n_iter} iterations"}
    Es, d, b, w = ph.spectrum(4, 60.0, 160.0, 95.0, 30.0, ph.BONE[0], ph.BONE[1], 80.0, 4000)
    l4 = O.Lines(Es, d, b, w, L=30.0, pixel=20e-6)
    per_px = []
    for j, (nx, ny) in enumerate(UNEVEN_SIZES):
        ells4 = ph.random_ellipsoids(band, nx, 20, 3.0, 40.0, margin=10.0, seed=4400 + j)
        t4 = ph.project_ellipsoids(ells4, band, nx, 20e-6)
        D4 = ph.poisson(O.forward(l4, t4), 1e4, 4500 + j)
        t0 = time.perf_counter()
        O.solve(l4, D4, n_iter=1, omega=0.4)
        per_px.append((time.perf_counter() - t0) / (band * nx))
    it_eq = float(np.mean(per_px)) * REF_PIX
    out["uneven_4line"] = {
        "sizes_nx_ny": [list(sz) for sz in UNEVEN_SIZES], "n_lines": 4,
        "s_per_2048sq_equiv_iteration": round(it_eq, 3),
        "equiv_2048sq_iterations_per_s": round(1.0 / it_eq, 4), "cores": 1,
        "sample": f"1 iteration on a {band}-row band of each size, scaled by pixel count "
                  f"(uniform size mix)"}
    return out


def cpu_baseline(n_it: int):
    """The FP64 oracle as it stands on the host cores, on a bounded sample of
    the headline workload: the first n_it of its 50 iterations, time scaled by
    50 / n_it (every iteration does the same work).  Timed on one thread, then
    as one such solve per core in separate processes (independent
    projections; the oracle itself is single threaded).  Returns the record
    and the data D it solved."""
    import multiprocessing as mp
    O, wl, ln, D = _oracle_workload()
    t1 = _oracle_sample(n_it, D)
    ncores = os.cpu_count() or 1
    with mp.get_context("spawn").Pool(ncores) as pool:
        t0 = time.perf_counter()
        pool.starmap(_oracle_sample, [(n_it, D)] * ncores)
        tn = time.perf_counter() - t0
    scale = wl.n_iter / n_it
    frac = wl.nx * wl.ny / REF_PIX
    single = frac / (t1 * scale)
    multi = ncores * frac / (tn * scale)
    rec = {"value": round(multi, 6), "unit": UNIT, "cores": ncores, "kind": "oracle",
           "cpu_model": _cpu_model(),
           "sample": f"{n_it} of {wl.n_iter} iterations of the 2048x2048 solve, scaled to the "
                     f"full solve; {ncores} independent solves, one per core in separate "
                     f"processes ({tn:.1f} s wall)",
           "single_thread": {"value": round(single, 6), "unit": UNIT, "cores": 1,
                             "sample": f"{n_it} of {wl.n_iter} iterations ({t1:.1f} s), scaled"},
           "other_configs": _oracle_other_configs()}
    return rec, D


def run_reference(a):
    """The oracle on the host cores, as the reference arm.  Each step is one
    iteration of the solve on a band of rows of the same workload, the band
    sized so the whole run takes about two minutes, scaled to 2048^2
    projections by pixel count and to 50 iterations."""
    rank, world, local = _dist()
    if rank != 0:
        return
    O, wl, ln, D = _oracle_workload()
    budget_s, full_iter_s = 120.0, 3.0
    per_step = budget_s / max(1, a.steps + a.warmup)
    rows = 16
    while rows * 2 <= wl.ny and full_iter_s * (rows * 2) / wl.ny <= per_step:
        rows *= 2
    y0 = (wl.ny - rows) // 2
    Db = np.ascontiguousarray(D[y0:y0 + rows])
    lnb = O.Lines(wl.energy_keV, wl.delta, wl.beta, wl.weights, wl.L, wl.pixel)
    T = np.zeros_like(Db)
    for _ in range(a.warmup):
        T, _ = O.solve(lnb, Db, T0=T, n_iter=1, omega=wl.omega)
    ts = []
    for _ in range(a.steps):
        t0 = time.perf_counter()
        T, _ = O.solve(lnb, Db, T0=T, n_iter=1, omega=wl.omega)
        ts.append(time.perf_counter() - t0)
    per_iter = float(np.mean(ts))
    per_solve = per_iter * wl.n_iter
    value = (rows * wl.nx / REF_PIX) / per_solve
    sample = (f"each step = 1 iteration on rows {y0}..{y0 + rows - 1} ({rows}x{wl.nx}) of the "
              f"2048x2048 workload (ms_per_step is that step), value scaled by pixel count and "
              f"by 50 iterations")
    out = {"metric": METRIC, "value": round(value, 6), "unit": UNIT, "n_gpus": world,
           "steps": a.steps, "warmup": a.warmup, "ms_per_step": round(per_iter * 1e3, 2),
           "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
           "data": "synthetic: seeded ellipsoid phantom, D = FP64 oracle forward + Poisson(1e4)",
           "config": bench_config(wl, world),
           "impl": "reference",
           "cpu_baseline": {"value": round(value, 6), "unit": UNIT, "cores": 1, "kind": "oracle",
                            "cpu_model": _cpu_model(), "sample": sample},
           "e2e": {"value": round(value, 6), "unit": UNIT, "h2d_bytes_per_step": 0,
                   "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


if __name__ == "__main__":
    args = _args()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)
