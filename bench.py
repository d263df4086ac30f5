"""Benchmark of the 3D LP step on GB300: particle-updates/s.

Workload: the 3D ideal-gas (gamma = 5/3) Gaussian gas cloud, 2,000,000 equal-mass
particles sampled from rho ~ exp(-r^2/0.1), p = rho^gamma, u = 0 (seeded,
synthetic).  One step = the whole hot path through the C ABI lp_step: bounding
cube, Morton keys, radix sort, gather, cell tables, neighbour query, CFL time
step on the device, fused GFD fits + Lax-Wendroff/upwind rates + estimator +
limiter blend + mover (FP32 fits, FP64 state, FP64 redo of ill-conditioned
stencils).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

Prints one JSON line.  --impl reference times the FP64 CPU oracle (the only
reference this paper has) on bounded samples of the same workload.
N > 1 (torchrun): independent replicas, one per GPU; no data-path collective.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "particle-updates/s (3D LP step) at 1e-5 rel err vs FP64; % HBM roofline"
UNIT = "particle-updates/s"
GAMMA = 5.0 / 3.0
KAPPA = 2.2
K_MAX = 64
CFL = 0.4
SEED = 4
WORKLOAD = "gas-cloud-3d-2M"
L2_FLUSH_BYTES = 256 << 20

# FP32 flops per particle of the fit + update pass as the kernels compute it
# (an FMA counts 2; a multiply, add, subtract or reciprocal 1), with N = 9
# unknowns, F = 5 fields, D = 3 axes and m neighbours:
#   central fit, per neighbour row: offsets and field differences from the hi/lo
#     records (2 subtractions and an add each: 3 D + 3 F), scaling (D), the nine
#     monomials (9), then the normal equations A^T A (45 FMA) and A^T B (N F = 45
#     FMA); once per particle the U^T D U factor (sum_k k (N - k) = 120 FMA, N
#     reciprocals, 36 multiplies) and the semi-normal solve of F right-hand
#     sides (2 x 36 F FMA, N reciprocals, N F multiplies);
#   correction pass, on the share of particles that ran it (the n_refined
#     counter): per row the row again, its residual (N F FMA) and A^T r (N F
#     FMA), then another semi-normal solve;
#   one-sided fits, on the share of particles that took the plain estimator:
#     2 D fits of k_side = 8 rows, each row built from its record (3 D + 3 F + D)
#     and rotated into a 3-unknown square-root-free Givens factor with F
#     right-hand sides (per column: 7; per later column 5; per right-hand side 5:
#     111 per row), plus a 3 x 3 back substitution of F right-hand sides per fit;
#   LW and UW rates, estimator, limiter, blend and mover: about 500.
FIT_N, FIT_F, FIT_D, FIT_KSIDE = 9, 5, 3, 8


def fit_flops_per_particle(m: float, refined_frac: float = 0.0, plain_frac: float = 1.0) -> float:
    N, F, D = FIT_N, FIT_F, FIT_D
    row = 3 * D + 3 * F + D + 9
    gram = 2 * (N * (N + 1) // 2 + N * F)
    factor = 2 * 120 + N + 36
    solve = 2 * (2 * 36 * F) + N + N * F
    central = m * (row + gram) + factor + solve
    correction = m * (row + 2 * 2 * N * F) + solve
    givens_row = (3 * D + 3 * F + D) + sum(7 + 5 * (D - 1 - k) + 5 * F for k in range(D))
    onesided = 2 * D * (FIT_KSIDE * givens_row + 2 * F * (D * (D - 1) // 2))
    return central + refined_frac * correction + plain_frac * onesided + 500.0


# DRAM bytes per particle of one fit pass (split schedule, FP32: k_step_central,
# k_step_central_refine, k_step_plain), measured by ncu (dram__bytes_read.sum +
# dram__bytes_write.sum, one pass, every launch of three timed steps) on the
# 2M-particle gas cloud this benchmark times: 2,118 MB per pass.  None when the
# kernels change and the figure has not been re-measured.
FIT_TRAFFIC_BPP_2M = 1058.8

# warp instructions per particle of one neighbour query (k_query_tile and the
# kernels over the groups and particles it leaves; smsp__inst_executed.sum from
# the same capture): the query is bound by instruction issue (integer, shuffle
# and shared-memory work), so it is reported against the SM issue peak of
# 4 warp instructions per clock per SM.
QUERY_INST_PP_2M = 914.0

# nominal FP64 rate of a GB300 (TFLOP/s): the roofline of the FP64 fit
FP64_PEAK_TFLOPS = 1.25

# algorithmic DRAM bytes per particle of the memory-bound phases
BYTES_PER_PARTICLE = {
    "grid+keys": 24 + 24 + 12,              # positions read (extent, keys), key + index write
    "radix-sort": 24,                       # per digit pass: key + index read and written once
    "gather": 76 + 76 + 64 + 32,            # state read; sorted copy, fit record and query positions written
    "cell-tables": 8 * 2,                   # sorted keys read (fill and clear)
}


def schedule_name(lp, sch: int) -> str:
    """The autotuner's choice as text: fit schedule + query schedule."""
    fit = ("split" if sch & lp.SCHED_SPLIT else "fused") + ("-queue" if sch & lp.SCHED_QUEUE_FIT else "")
    query = "query-warp" if sch & lp.SCHED_QUERY_WARP else (
        "query-tiles-queue" if sch & lp.SCHED_QUEUE_QUERY else "query-tiles")
    return fit + "+" + query


def parse(argv=None):
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=20)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--particles", type=int, default=None,
                    help="particles (default: 2M for the gas cloud, about 8M for the jet snapshot)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--cpu-seconds", type=float, default=12.0)
    ap.add_argument("--workload", default="gas-cloud", choices=["gas-cloud", "jet-snapshot", "kh-ensemble", "jet-inflow"],
                    help="jet-snapshot: the static jet-shaped state (density ratio 1e3, gamma 1.4); jet-inflow: the "
                         "jet grown through a reservoir inlet to --particles (default 8M), then timed")
    ap.add_argument("--sims", type=int, default=256)
    ap.add_argument("--density-ratio", type=float, default=1e3,
                    help="jet-inflow: jet / ambient density ratio")
    ap.add_argument("--select", default="octant", choices=["nearest", "octant"],
                    help="neighbours kept beyond k_max (the jet workloads; the gas cloud keeps the nearest): "
                         "octant-balanced (the default: with the nearest only, the ambient particles next to the "
                         "jet lose their one-sided stencils, and the jet's volumes and radii blow up within a few "
                         "steps), or the nearest")
    ap.add_argument("--limiter", default="flagged", choices=["flagged", "uw"],
                    help="jet-inflow: the limiter mode")
    ap.add_argument("--grow-seconds", type=float, default=240.0,
                    help="jet-inflow: wall-time budget of the untimed growth phase")
    ap.add_argument("--estimator", default="plain", choices=["plain", "mlp"],
                    help="mlp: train the learned estimator on this workload's own plain steps, then time "
                         "steps gated by it")
    ap.add_argument("--no-autotune", action="store_true")
    ap.add_argument("--eager", action="store_true",
                    help="time the steps as separate lp_step calls instead of replaying a captured step")
    ap.add_argument("--schedule", default=None, choices=["fused", "split"],
                    help="fit schedule to time (instead of the autotuner's choice)")
    ap.add_argument("--no-forms", action="store_true",
                    help="skip the FP64 and learned-estimator forms reported beside the headline")
    ap.add_argument("--precision", default="fp32", choices=["fp32", "fp64"],
                    help="fp64: every fit and rate in FP64 (the plain FP64 GPU form)")
    ap.add_argument("--compare-estimators", type=int, default=0, metavar="STEPS",
                    help="gas cloud: advance the same state STEPS steps with the plain and with the learned "
                         "estimator (the learned run takes the plain run's CFL steps) and report both times "
                         "and the learned run's drift from the plain one")
    return ap.parse_args(argv)


def max_over_ranks(values, world, torch, dist, device):
    """Each value's maximum over the ranks: the job takes as long as its
    slowest rank."""
    t = torch.tensor([float(v) for v in values], dtype=torch.float64, device=device)
    if world > 1:
        dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return [float(v) for v in t]


def job_rate(world, n, steps, ms):
    """Particle-updates per second of the whole job: each of the world ranks
    advances its own n particles per step (replicas)."""
    return world * n * steps / (ms * 1e-3)


def fit_traffic(precision, estimator, split, workload, n, bpp=None):
    """DRAM bytes of one fit pass from an ncu figure per particle, or None where
    no capture describes the pass: the figure is of the split schedule's FP32
    kernels with the plain estimator on the gas cloud."""
    if precision == "fp32" and estimator == "plain" and split and workload == "gas-cloud" and bpp:
        return bpp * n
    return None


def dist_info():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


# the single-simulation 3D workloads: generator, gamma, default size, k_max
# (the jet's neighbour counts run from 20 to 80)
WORKLOADS = {"gas-cloud": ("gas-cloud-3d", 5.0 / 3.0, 2_000_000, 64),
             "jet-snapshot": ("jet-snapshot-3d", 1.4, 8_000_000, 80),
             "jet-inflow": ("jet-inflow-3d", 1.4, 8_000_000, 80)}
ACTIVE = "gas-cloud"
SELECT = "nearest"            # neighbours kept beyond k_max: the jet workloads take --select


def select_workload(args):
    """Set the workload's gamma and name, and its default size."""
    global ACTIVE, GAMMA, WORKLOAD, K_MAX, SELECT
    if args.workload in WORKLOADS:
        ACTIVE = args.workload
    name, GAMMA, n0, K_MAX = WORKLOADS[ACTIVE]
    SELECT = args.select if ACTIVE != "gas-cloud" else "nearest"
    if args.particles is None:
        args.particles = n0
    WORKLOAD = name


def size_tag(n):
    return ("%dM" % (n // 1_000_000)) if n % 1_000_000 == 0 else (
        "%.2fM" % (n / 1e6) if n >= 1_000_000 else "%dk" % round(n / 1e3))


def workload_state(n, seed=SEED):
    global WORKLOAD
    from paper_2206_11998_gb300 import inputs
    if ACTIVE == "jet-snapshot":
        st = inputs.jet_snapshot_3d(n, seed=seed + 6)
    else:
        st = inputs.gas_cloud_3d(n, seed=seed, gamma=GAMMA)
    WORKLOAD = WORKLOADS[ACTIVE][0] + "-" + size_tag(st["V"].shape[0])
    return st


def config_dict(n, extra=None):
    d = {"workload": WORKLOAD, "particles": n, "dim": 3, "gamma": GAMMA, "kappa": KAPPA, "k_max": K_MAX,
         "select": SELECT, "cfl": CFL, "limiter": "flagged", "precision": "FP32 fits + FP64 state, FP64 redo",
         "l2": "flushed between timed steps (256 MiB write); inputs also exceed L2",
         "parallelism": "replicas"}
    if extra:
        d.update(extra)
    return d


# ---------------------------------------------------------------------------
# CPU oracle timing
# ---------------------------------------------------------------------------

def cpu_model():
    """The host CPU's model name (lscpu, else /proc/cpuinfo, else the machine type)."""
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.lower().startswith("model name"):
                return line.split(":", 1)[1].strip()
    except Exception:
        pass
    try:
        for line in open("/proc/cpuinfo"):
            if line.lower().startswith(("model name", "cpu model")):
                return line.split(":", 1)[1].strip()
    except OSError:
        pass
    import platform
    return platform.machine()


def oracle_sample_rate(state, target_s, seed=0, threads=None):
    """Time the oracle's step on a bounded random sample of the workload's
    particles (full state visible), on all host cores or on `threads`.
    Returns (updates/s, cores used, sample size, seconds)."""
    import oracle
    oracle.build()
    if threads:
        saved = oracle.num_threads()
        oracle.set_num_threads(threads)
        try:
            return oracle_sample_rate(state, target_s, seed)
        finally:
            oracle.set_num_threads(saved)
    from paper_2206_11998_gb300 import inputs
    cfg = oracle.make_config(3, gamma=GAMMA, radius_mode=oracle.RADIUS_VOLUME, kappa=KAPPA, k_max=K_MAX,
                             k_side=8, limiter=oracle.LIM_FLAGGED, s_ref=inputs.field_scales(state),
                             select=oracle.SELECT_OCTANT if SELECT == "octant" else oracle.SELECT_NEAREST)
    n = state["V"].shape[0]
    rng = np.random.default_rng(seed)
    q0 = np.sort(rng.choice(n, 256, replace=False))
    t0 = time.perf_counter()
    oracle.step(cfg, state, 1e-4, query=q0)
    t1 = time.perf_counter() - t0
    q_n = int(min(n, max(256, 256 * target_s / max(t1, 1e-3))))
    q = np.sort(rng.choice(n, q_n, replace=False))
    t0 = time.perf_counter()
    oracle.step(cfg, state, 1e-4, query=q)
    dt = time.perf_counter() - t0
    cores = oracle.num_threads()
    return q_n / dt, cores, q_n, dt


# ---------------------------------------------------------------------------
# clocks
# ---------------------------------------------------------------------------

class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.proc = None
        self.gpu = gpu_index
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(prefix="lp_clocks_", suffix=".csv")
            self.f = os.fdopen(fd, "w")
            cmd = ["nvidia-smi", "--query-gpu=" + self.FIELDS, "--format=csv,noheader,nounits", "-lms", "50"]
            if self.gpu is not None:
                cmd += ["-i", str(self.gpu)]
            self.proc = subprocess.Popen(cmd, stdout=self.f, stderr=subprocess.DEVNULL)
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
        try:
            os.unlink(self.path)
        except OSError:
            pass
        if not sm:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        return {"sm_mhz": statistics.median(sm), "sm_max_mhz": max(smax), "reasons": sorted(reasons),
                "samples": len(sm)}


def gpu_index_for(local_rank):
    vis = os.environ.get("CUDA_VISIBLE_DEVICES")
    if vis:
        ids = [v for v in vis.split(",") if v.strip()]
        if local_rank < len(ids) and ids[local_rank].strip().isdigit():
            return int(ids[local_rank])
    return local_rank


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        try:
            return json.load(open(p)), "measured"
        except Exception:
            pass
    return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "sm_max_mhz": 2070.0}, "fallback"


# ---------------------------------------------------------------------------
# the GPU arm
# ---------------------------------------------------------------------------

def run_ours(args):
    import torch
    import torch.distributed as dist

    from paper_2206_11998_gb300 import build as b
    from paper_2206_11998_gb300 import inputs, lp

    rank, world, local = dist_info()
    if world > 1:
        dist.init_process_group("nccl", rank=rank, world_size=world)
    torch.cuda.set_device(local)
    b.build()
    state = workload_state(args.particles, seed=SEED + rank)
    n = state["V"].shape[0]
    stream = torch.cuda.Stream()
    mlp_info = None
    kw = {}
    if args.estimator == "mlp":
        params, mlp_info = train_gate(lp, inputs, state, n, stream, torch)
        kw = dict(estimator=lp.EST_MLP, mlp_tau_lo=mlp_info["tau_lo"])
    prec = lp.PREC_FP64 if args.precision == "fp64" else lp.PREC_FP32
    if SELECT == "octant":
        kw["select"] = lp.SELECT_OCTANT
    cfg = lp.make_config(3, n, precision=prec, radius_mode=lp.RADIUS_VOLUME, kappa=KAPPA, k_max=K_MAX,
                         k_side=8, gamma=GAMMA, limiter=lp.LIM_FLAGGED, s_ref=inputs.field_scales(state), **kw)
    ctx = lp.Context(cfg)
    if args.estimator == "mlp":
        ctx.mlp_set_params(params)
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")

    def barrier():
        torch.cuda.synchronize()
        if world > 1:
            dist.barrier()
        torch.cuda.synchronize()

    with torch.cuda.stream(stream):
        ps = lp.ParticleSet.from_state(state)
        t_dev = torch.zeros(1, dtype=torch.float64, device="cuda")
        for _ in range(args.warmup):
            ctx.step(ps, dt=0.0, cfl=CFL, t=t_dev, stream=stream)
        tune = None
        if args.schedule:
            ctx.set_schedule({"fused": lp.SCHED_FUSED, "split": lp.SCHED_SPLIT}[args.schedule])
        elif not args.no_autotune:
            tune = ctx.autotune(ps, dt=0.0, cfl=CFL, reps=3, stream=stream)
            sch = ctx.schedule()
            tune["chosen"] = schedule_name(lp, sch)
        # mean neighbour count of the current lists (algorithmic work per particle)
        cnt = ctx.export_neighbors(n, stream=stream)[0]
        m_mean = float(cnt.double().mean().item())
        stream.synchronize()
        # the timed steps replay one captured step (lp_graph_capture / lp_graph_launch):
        # the same kernels with no host launch between them
        graph = not args.eager
        if graph:
            ctx.graph_capture(ps, dt=0.0, cfl=CFL, t=t_dev, stream=stream)
            for _ in range(2):
                ctx.graph_launch(stream=stream)
            stream.synchronize()
        ctx.reset_stats(stream=stream)
        launches0 = ctx.stats(stream=stream)["kernel_launches"]
        sampler = ClockSampler(gpu_index_for(local))
        barrier()
        sampler.start()
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
        wall0 = time.perf_counter()
        marked = nvtx_push("timed_steps", torch)      # lets ncu list the timed launches alone
        for k in range(args.steps):
            flush.zero_()
            ev[k][0].record(stream)
            if graph:
                ctx.graph_launch(stream=stream)
            else:
                ctx.step(ps, dt=0.0, cfl=CFL, t=t_dev, stream=stream)
            ev[k][1].record(stream)
        stream.synchronize()
        if marked:
            torch.cuda.nvtx.range_pop()
        wall = time.perf_counter() - wall0
        barrier()
        clocks = sampler.stop()
        st = ctx.stats(stream=stream)
        launches = st["kernel_launches"] - launches0
        step_ms = [a.elapsed_time(bb) for a, bb in ev]
        total_ms = sum(step_ms)
        # the per-phase split, from as many eager steps with phase events (which
        # a graph cannot hold), after the timed ones
        ctx.phase_times(stream=stream)
        ctx.set_profiling(True)
        for _ in range(args.steps):
            flush.zero_()
            ctx.step(ps, dt=0.0, cfl=CFL, t=t_dev, stream=stream)
        ctx.set_profiling(False)
        phases = ctx.phase_times(stream=stream)

        if mlp_info is not None:
            mlp_info.update(audit_gate(lp, inputs, ps, n, cfg, params, stream, torch))
            mlp_info["skipped_per_step"] = st["n_mlp_skip"] / args.steps

        # end to end through the same C-ABI call with host buffers
        e2e = run_e2e(ctx, state, n, args, stream, lp, torch, flush)

        # the plain FP64 GPU form and the FP32 + learned form of the same step
        forms = None
        if world == 1 and not args.no_forms and args.precision == "fp32" and args.estimator == "plain":
            forms = other_forms(args, state, n, stream, lp, inputs, torch, flush)
            try:
                del ps
                r = ensemble_measure(args, args.sims, min(args.steps, 10), args.warmup)
                forms["fp32_batched_kh_ensemble"] = {
                    "workload": "kh-ensemble-%d: 2D periodic shear layers of U[10k, 200k] particles" % r["sims"],
                    "particles": r["particles"], "ms_per_step": r["batched_ms"],
                    "value": r["particles"] / (r["batched_ms"] * 1e-3), "steps": r["steps"],
                    "form": "every simulation in one lp_step_batched per step, replayed from a captured CUDA graph",
                    "unbatched_ms_per_step": r["loop_ms"], "speedup_vs_unbatched": r["loop_ms"] / r["batched_ms"],
                    "launches_per_step": r["launches"] / r["steps"], "autotune": r["tune"]}
            except Exception as exc:
                forms["ensemble_error"] = repr(exc)

    total_ms, e2e_ms = max_over_ranks([total_ms, e2e["ms"]], world, torch, dist, "cuda")
    value = job_rate(world, n, args.steps, total_ms)
    e2e_value = job_rate(world, n, args.steps, e2e_ms)

    peaks, peak_kind = measured_peaks()
    sm_max = float(peaks.get("sm_max_mhz", 2070.0))
    n_sm = torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count
    fp32_peak = n_sm * 128 * 2 * sm_max * 1e6 / 1e12      # TFLOP/s, FP32 CUDA cores
    hbm_peak = float(peaks.get("hbm_gbs", 6800.0))
    per_phase = {}
    for name, (ms, nl) in phases.items():
        if nl == 0 and ms == 0.0:
            continue
        entry = {"ms_per_step": ms / args.steps, "launches": nl, "share": ms / max(1e-9, sum(v[0] for v in phases.values()))}
        if name in BYTES_PER_PARTICLE:
            # the sort runs three kernels per digit pass
            passes = nl / (3 * args.steps) if name == "radix-sort" else 1
            byts = BYTES_PER_PARTICLE[name] * n * passes
            gbs = byts / (ms / args.steps * 1e-3) / 1e9 if ms > 0 else None
            entry.update({"bound": "hbm", "achieved_gbs": gbs, "frac_of_hbm": gbs / hbm_peak if gbs else None})
        per_phase[name] = entry
    fit_phase = "fit+update" if args.precision == "fp32" else "fit+update-fp64"
    fit_ms = phases[fit_phase][0] / args.steps          # one fit pass over all n particles
    refined_frac = st["n_refined"] / (n * args.steps)
    plain_frac = 1.0 - st["n_mlp_skip"] / (n * args.steps)
    fpp = fit_flops_per_particle(m_mean, refined_frac if args.precision == "fp32" else 0.0, plain_frac)
    flops = fpp * n
    achieved = flops / (fit_ms * 1e-3) / 1e12
    dominant = max(per_phase, key=lambda k: per_phase[k]["ms_per_step"])
    sched = ctx.schedule()
    fit_kernels = ("k_step_central + k_step_plain" if sched & lp.SCHED_SPLIT else "k_step") + \
        ("<float,3>" if args.precision == "fp32" else "<double,3>")
    # the captured figure is of the launch-grid split kernels (the persistent
    # ones read and write the same data, but were not captured)
    traffic = fit_traffic(args.precision, args.estimator,
                          bool(sched & lp.SCHED_SPLIT) and not (sched & lp.SCHED_QUEUE_FIT), ACTIVE, n,
                          FIT_TRAFFIC_BPP_2M if n == 2_000_000 else None)
    if args.precision == "fp32":
        alu_peak = fp32_peak
        alu_source = "FP32 CUDA cores: %d SM x 128 lanes x 2 x %.0f MHz (%s max clock)" % (n_sm, sm_max, peak_kind)
    else:
        alu_peak = FP64_PEAK_TFLOPS
        alu_source = "nominal GB300 FP64 rate (the FP64 fit runs on the FP64 units)"
    roofline = {"kernel": fit_kernels + " (fit+update pass)", "dominant_phase": dominant, "bound": "alu",
                "achieved": achieved, "peak": alu_peak, "unit": "TFLOP/s", "frac": achieved / alu_peak,
                "peak_source": alu_source,
                "flops_per_particle": fpp, "flop_model": "the operations the kernels run: normal equations, "
                "U^T D U factor and solve; correction pass on the refined share; one-sided Givens fits on the "
                "plain-estimator share", "mean_neighbors": m_mean, "refined_frac": refined_frac,
                "plain_frac": plain_frac, "traffic": traffic,
                "traffic_source": "ncu dram__bytes_read.sum + dram__bytes_write.sum of the fit kernels, every launch "
                                  "of three timed steps of this 2M workload"
                                  if traffic else None,
                "limiter": "not the FP32 pipe: the L1 data pipe's wavefronts for the per-lane gathers of neighbour "
                           "records (ncu, 400k cloud: 76% of peak in k_step_central, 69% in k_step_plain) and the "
                           "latency of those loads (long_scoreboard the top stall)"}
    query_roofline = None
    if ("neighbor-query" in phases and phases["neighbor-query"][0] > 0 and n == 2_000_000
            and ACTIVE == "gas-cloud" and not (sched & lp.SCHED_QUERY_WARP)):
        q_ms = phases["neighbor-query"][0] / args.steps
        issue_peak = n_sm * 4 * sm_max * 1e6
        q_ach = QUERY_INST_PP_2M * n / (q_ms * 1e-3)
        tile_kernel = "k_query_tile_q (work queue)" if sched & lp.SCHED_QUEUE_QUERY else "k_query_tile"
        query_roofline = {"kernel": tile_kernel + " + k_query_groups + k_query_left (neighbour query)", "bound": "issue",
                          "achieved": q_ach, "peak": issue_peak, "unit": "warp instructions/s",
                          "frac": q_ach / issue_peak, "inst_per_particle": QUERY_INST_PP_2M,
                          "peak_source": "%d SM x 4 schedulers x 1 warp instruction per clock x %.0f MHz" % (n_sm, sm_max),
                          "inst_source": "ncu smsp__inst_executed.sum, every launch of three timed steps of this workload"}
    cpu = None
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        rate, cores, q_n, secs = oracle_sample_rate(state, args.cpu_seconds)
        rate1, _, q1, secs1 = oracle_sample_rate(state, max(2.0, args.cpu_seconds / 4), seed=1, threads=1)
        cpu = {"value": rate, "unit": UNIT, "cores": cores, "kind": "oracle", "cpu_model": cpu_model(),
               "single_thread": {"value": rate1, "unit": UNIT, "cores": 1,
                                 "sample": "oracle step of %d random particles, %.1f s" % (q1, secs1)},
               "sample": "oracle step of %d random particles of the %s cloud (full state visible), %.1f s"
                         % (q_n, size_tag(n), secs)}
    if rank == 0:
        line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
                "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
                "scaling": "weak", "vs_baseline": None, "dtype": "f32" if args.precision == "fp32" else "f64",
                "data": "synthetic",
                "config": config_dict(n, {"fit_ms_per_step": fit_ms, "wall_s_timed": wall,
                                          "precision": ("FP32 fits + FP64 state, FP64 redo" if args.precision == "fp32"
                                                        else "FP64 fits, rates and state"),
                                          "flagged_per_step": st["n_flagged"] / args.steps,
                                          "fp64_redo_per_step": st["n_fp64_redo"] / args.steps,
                                          "fit_schedule": tune, "estimator": args.estimator,
                                          "learned_gate": mlp_info,
                                          "execution": ("one captured lp_step replayed per timed step (lp_graph_launch); "
                                                        "phases from as many eager steps with phase events"
                                                        if graph else "one lp_step call per timed step")}),
                "roofline": roofline, "query_roofline": query_roofline, "cpu_baseline": cpu,
                "e2e": {"value": e2e_value, "unit": UNIT, "h2d_bytes_per_step": e2e["h2d"],
                        "d2h_bytes_per_step": e2e["d2h"],
                        "api": "lp_step_host on page-locked host arrays (state copied in; the new state "
                               "written into the host arrays by the step's kernels)"},
                "gpu_launches": launches, "clocks": clocks, "phases": per_phase, "forms": forms}
        print(json.dumps(line), flush=True)
    ctx.close()
    if world > 1:
        dist.destroy_process_group()


MLP_MISS = 0.01   # share of the training set's flags the gate threshold may clear


def train_gate(lp, inputs, state, n, stream, torch):
    """Train the learned estimator on features and plain-estimator flags of two
    plain steps of this workload (untimed): returns (parameters, info)."""
    cfg = lp.make_config(3, n, precision=lp.PREC_FP32, kappa=KAPPA, k_max=K_MAX, gamma=GAMMA,
                         s_ref=inputs.field_scales(state))
    c0 = lp.Context(cfg)
    X, y = [], []
    with torch.cuda.stream(stream):
        ps = lp.ParticleSet.from_state(state)
        for _ in range(2):
            f = torch.empty((n, 8), dtype=torch.float32, device="cuda")
            g = torch.empty(n, dtype=torch.uint8, device="cuda")
            c0.step(ps, dt=0.0, cfl=CFL, features=f, flag=g, stream=stream)
            X.append(f)
            y.append(g.float())
        X = torch.cat(X)
        y = torch.cat(y)
        gen = torch.Generator(device="cuda").manual_seed(0)
        perm = torch.randperm(X.shape[0], device="cuda", generator=gen)
        X, y = X[perm].contiguous(), y[perm].contiguous()
        pos = float((y == 0).sum()) / max(1.0, float((y == 1).sum()))
        c0.mlp_set_params(lp.mlp_init_params(1))
        t0 = time.perf_counter()
        losses = c0.mlp_train(X, y, epochs=20, batch=8192, lr=1e-2, pos_weight=pos, stream=stream)
        stream.synchronize()
        secs = time.perf_counter() - t0
        params = c0.mlp_get_params()[0]
        # threshold calibrated on the training set: MLP_MISS of its flags fall below it
        p = c0.mlp_infer(X, stream=stream)
        tau = float(torch.quantile(p[y > 0.5].float(), MLP_MISS).item())
    c0.close()
    return params, {"train_samples": int(X.shape[0]), "train_epochs": 20, "train_s": secs,
                    "loss_first": float(losses[0]), "loss_last": float(losses[-1]), "tau_lo": tau,
                    "calibrated_miss": MLP_MISS}


def other_forms(args, state, n, stream, lp, inputs, torch, flush):
    """The plain FP64 GPU form and the FP32 + learned-estimator form of the
    headline's step on the same workload, timed like it (L2 flushed between
    steps, CUDA events on the stream), and the one-step error of each FP32 form
    against the FP64 form from the same initial state with the same dt.  The
    FP64 form is itself within 1e-12 of the FP64 oracle in the parity tests."""
    sref = inputs.field_scales(state)
    base = dict(radius_mode=lp.RADIUS_VOLUME, kappa=KAPPA, k_max=K_MAX, k_side=8, gamma=GAMMA,
                limiter=lp.LIM_FLAGGED, s_ref=sref)
    out = {}

    def timed(ctx, steps, warmup, graph=False):
        ps = lp.ParticleSet.from_state(state)
        for _ in range(warmup):
            ctx.step(ps, dt=0.0, cfl=CFL, stream=stream)
        if graph:
            ctx.graph_capture(ps, None, 1, dt=0.0, cfl=CFL, stream=stream)
            ctx.graph_launch(stream=stream)
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
        for k in range(steps):
            flush.zero_()
            ev[k][0].record(stream)
            if graph:
                ctx.graph_launch(stream=stream)
            else:
                ctx.step(ps, dt=0.0, cfl=CFL, stream=stream)
            ev[k][1].record(stream)
        stream.synchronize()
        return sum(a.elapsed_time(b) for a, b in ev) / steps

    def one_step(ctx, dt):
        ps = lp.ParticleSet.from_state(state)
        ctx.reset_stats(stream=stream)
        ctx.step(ps, dt=dt, cfl=CFL, stream=stream)
        stream.synchronize()
        idx = ps.id.long()
        byid = lambda t: torch.empty_like(t).index_copy_(0, idx, t)
        return {"V": byid(ps.V), "P": byid(ps.P), "u": [byid(a) for a in ps.u]}, ctx.stats(stream=stream)

    s0 = {"V": torch.as_tensor(state["V"], device="cuda"), "P": torch.as_tensor(state["P"], device="cuda"),
          "u": [torch.as_tensor(a, device="cuda") for a in state["u"]]}

    def errors(g, o, dt):
        e = {}
        for nm, a, b, z in [("V", g["V"], o["V"], s0["V"]), ("P", g["P"], o["P"], s0["P"])] + [
                ("u%d" % k, g["u"][k], o["u"][k], s0["u"][k]) for k in range(3)]:
            d = float((a - b).abs().max())
            e[nm] = d / max(float(b.abs().max()), 1e-300)
            e["rate_" + nm] = d / max(float((b - z).abs().max()), 1e-300)
        return e

    try:
        c64 = lp.Context(lp.make_config(3, n, precision=lp.PREC_FP64, **base))
        ref, st64 = one_step(c64, 0.0)
        dt = st64["dt"]
        k64 = max(2, min(args.steps, 3))
        ms64 = timed(c64, k64, 1)
        c64.close()
        out["fp64"] = {"ms_per_step": ms64, "value": n / (ms64 * 1e-3), "steps": k64, "dtype": "f64",
                       "form": "every fit, rate and the state in FP64 on the GPU"}
        c32 = lp.Context(lp.make_config(3, n, precision=lp.PREC_FP32, **base))
        g32, _ = one_step(c32, dt)
        c32.close()
        out["accuracy_vs_fp64_form"] = {"fp32": errors(g32, ref, dt), "dt": dt,
                                        "note": "one step from the initial state with the FP64 form's CFL dt; "
                                                "per field max|a - b| / max|b| for the state, and for the "
                                                "rates (s^{n+1} - s^n)/dt"}
    except Exception as exc:                                  # reported, never fatal to the headline
        out["fp64_error"] = repr(exc)
        ref = None
    try:
        params, info = train_gate(lp, inputs, state, n, stream, torch)
        cm = lp.Context(lp.make_config(3, n, precision=lp.PREC_FP32, estimator=lp.EST_MLP,
                                       mlp_tau_lo=info["tau_lo"], **base))
        cm.mlp_set_params(params)
        if ref is not None:
            gm, stm = one_step(cm, dt)
            out["accuracy_vs_fp64_form"]["fp32_learned"] = errors(gm, ref, dt)
            info["skipped"] = stm["n_mlp_skip"]
        ms_e = timed(cm, args.steps, args.warmup)
        ms_g = timed(cm, args.steps, 1, graph=True)
        cm.close()
        cfg = lp.make_config(3, n, precision=lp.PREC_FP32, estimator=lp.EST_MLP, mlp_tau_lo=info["tau_lo"], **base)
        ps = lp.ParticleSet.from_state(state)
        info.update(audit_gate(lp, inputs, ps, n, cfg, params, stream, torch))
        del ps
        out["fp32_learned"] = {"ms_per_step": ms_g, "value": n / (ms_g * 1e-3), "steps": args.steps,
                               "eager_ms_per_step": ms_e, "dtype": "f32",
                               "form": "FP32 fits, learned state estimator (plain estimator as fallback), "
                                       "the step replayed from a captured CUDA graph",
                               "learned_gate": info}
    except Exception as exc:
        out["learned_error"] = repr(exc)
    return out


def audit_gate(lp, inputs, ps, n, cfg, params, stream, torch):
    """One audited step from a copy of the current state: flags the learned gate
    cleared that the plain estimator raises."""
    cfg.mlp_audit = 1
    ca = lp.Context(cfg)
    ca.mlp_set_params(params)
    cp = lp.ParticleSet(x=[a.clone() for a in ps.x], V=ps.V.clone(), u=[a.clone() for a in ps.u], P=ps.P.clone(),
                        m=ps.m.clone(), id=ps.id.clone())
    ca.step(cp, dt=0.0, cfl=CFL, stream=stream)
    st = ca.stats(stream=stream)
    ca.close()
    cfg.mlp_audit = 0
    return {"audit_skipped": st["n_mlp_skip"], "audit_missed_flags": st["n_mlp_miss"],
            "audit_flagged": st["n_flagged"]}


def nvtx_push(name, torch):
    try:
        torch.cuda.nvtx.range_push(name)
        return True
    except Exception:
        return False


def run_e2e(ctx, state, n, args, stream, lp, torch, flush):
    """Each step through lp_step_host on page-locked host arrays: the host ->
    device copy of the whole state (part of it overlapping the key sort) and
    the new state written back into the host arrays by the step's kernels,
    all inside the timed region."""
    hps = lp.ParticleSet.from_state_host(state)
    arrays = list(hps.x) + [hps.V] + list(hps.u) + [hps.P, hps.m, hps.id]
    h2d = sum(v.numel() * v.element_size() for v in arrays)
    d2h = h2d
    with torch.cuda.stream(stream):
        for _ in range(max(1, min(args.warmup, 2))):
            ctx.step_host(hps, dt=0.0, cfl=CFL, stream=stream)
        stream.synchronize()
        steps = max(1, min(args.steps, 10))
        evs = []
        for _ in range(steps):
            flush.zero_()
            a = torch.cuda.Event(enable_timing=True)
            b2 = torch.cuda.Event(enable_timing=True)
            a.record(stream)
            ctx.step_host(hps, dt=0.0, cfl=CFL, stream=stream)
            b2.record(stream)
            evs.append((a, b2))
        stream.synchronize()
    ms = sum(a.elapsed_time(b2) for a, b2 in evs) / steps * args.steps
    return {"ms": ms, "h2d": h2d, "d2h": d2h}


# ---------------------------------------------------------------------------
# the reference arm: the FP64 CPU oracle
# ---------------------------------------------------------------------------

def run_reference(args):
    rank, world, local = dist_info()
    if rank != 0:
        return
    state = workload_state(args.particles)
    n = state["V"].shape[0]
    import oracle
    oracle.build()
    from paper_2206_11998_gb300 import inputs
    cfg = oracle.make_config(3, gamma=GAMMA, radius_mode=oracle.RADIUS_VOLUME, kappa=KAPPA, k_max=K_MAX,
                             k_side=8, limiter=oracle.LIM_FLAGGED, s_ref=inputs.field_scales(state),
                             select=oracle.SELECT_OCTANT if SELECT == "octant" else oracle.SELECT_NEAREST)
    rng = np.random.default_rng(1)
    # size one step's sample so that the whole run stays within a few minutes
    budget_s = 150.0
    probe = np.sort(rng.choice(n, 128, replace=False))
    t0 = time.perf_counter()
    oracle.step(cfg, state, 1e-4, query=probe)
    per = (time.perf_counter() - t0) / 128
    q_n = int(max(64, min(n, budget_s / max(1, args.steps + args.warmup) / max(per, 1e-7))))
    times = []
    for k in range(args.warmup + args.steps):
        q = np.sort(rng.choice(n, q_n, replace=False))
        t0 = time.perf_counter()
        oracle.step(cfg, state, 1e-4, query=q)
        if k >= args.warmup:
            times.append(time.perf_counter() - t0)
    ms = 1e3 * sum(times) / len(times)
    value = q_n / (ms * 1e-3)
    cores = oracle.num_threads()
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": config_dict(n, {"reference": "FP64 CPU oracle (oracle/lp_oracle.c), OpenMP", "precision": "FP64 (oracle)"}),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores, "kind": "oracle",
                             "sample": "per step: oracle step of %d random particles of the 2M cloud" % q_n},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------------------
# the batched ensemble: many independent 2D shear layers in one step
# ---------------------------------------------------------------------------

KH_GAMMA = 1.4


def kh_states(nsim):
    from paper_2206_11998_gb300 import inputs
    sizes = inputs.kh_ensemble_sizes(nsim)
    amps = inputs.kh_ensemble_amplitudes(nsim)
    return [inputs.kh_2d(int(sizes[k]), float(amps[k]), seed=1000 + k) for k in range(nsim)]


def kh_cfg(lp, n, nsim):
    return lp.make_config(2, n, precision=lp.PREC_FP32, kappa=KAPPA, k_max=40, gamma=KH_GAMMA, periodic=(1, 1, 0),
                          box_lo=(0, 0, 0), box_hi=(1, 1, 1), s_ref=(1.0, 0.5, 0.5, 2.5), max_sims=nsim,
                          max_level=8)


def ensemble_measure(args, nsim, steps, warmup):
    """Batched: all simulations in one lp_step_batched, replayed from a CUDA
    graph.  Unbatched comparison: one lp_step per simulation, each with its own
    context, in a loop.  Returns the measurements (dict)."""
    import torch

    from paper_2206_11998_gb300 import build as b
    from paper_2206_11998_gb300 import lp

    b.build()
    sims = kh_states(nsim)
    sizes = np.array([s["V"].shape[0] for s in sims])
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    n = int(offs[-1])
    st = {k: np.concatenate([s[k] for s in sims]) for k in ("V", "P", "m")}
    st["x"] = [np.concatenate([s["x"][a] for s in sims]) for a in range(2)]
    st["u"] = [np.concatenate([s["u"][a] for s in sims]) for a in range(2)]
    st["id"] = np.arange(n, dtype=np.uint32)
    ctx = lp.Context(kh_cfg(lp, n, nsim))
    stream = torch.cuda.Stream()
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
    with torch.cuda.stream(stream):
        ps = lp.ParticleSet.from_state(st)
        offs_d = torch.as_tensor(offs, device="cuda")
        t = torch.zeros(nsim, dtype=torch.float64, device="cuda")
        ctx.step_batched(ps, offs_d, nsim, dt=0.0, cfl=CFL, t=t, stream=stream)
        tune = None
        if not args.no_autotune:
            tune = ctx.autotune(ps, offs_d, nsim, dt=0.0, cfl=CFL, reps=2, stream=stream)
            sch = ctx.schedule()
            tune["chosen"] = schedule_name(lp, sch)
        ctx.graph_capture(ps, offs_d, nsim, dt=0.0, cfl=CFL, t=t, stream=stream)
        for _ in range(warmup):
            ctx.graph_launch(stream=stream)
        stream.synchronize()
        l0 = ctx.stats(stream=stream)["kernel_launches"]
        sampler = ClockSampler(gpu_index_for(0))
        sampler.start()
        ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
        for k in range(steps):
            flush.zero_()
            ev[k][0].record(stream)
            ctx.graph_launch(stream=stream)
            ev[k][1].record(stream)
        stream.synchronize()
        clocks = sampler.stop()
        launches = ctx.stats(stream=stream)["kernel_launches"] - l0
        batched_ms = sum(a.elapsed_time(bb) for a, bb in ev) / steps
        # per-phase times of one eager batched step
        ctx.phase_times(stream=stream)
        ctx.set_profiling(True)
        ctx.step_batched(ps, offs_d, nsim, dt=0.0, cfl=CFL, t=t, stream=stream)
        phases = ctx.phase_times(stream=stream)
        ctx.set_profiling(False)
    ctx.close()
    del ps
    # unbatched: one context per simulation, one lp_step each, in a loop
    with torch.cuda.stream(stream):
        ctxs, pss = [], []
        for s in sims:
            c = lp.Context(kh_cfg(lp, s["V"].shape[0], 1))
            ctxs.append(c)
            pss.append(lp.ParticleSet.from_state(s))
        for c, p in zip(ctxs, pss):
            c.step(p, dt=0.0, cfl=CFL, stream=stream)
        stream.synchronize()
        a = torch.cuda.Event(enable_timing=True)
        bb = torch.cuda.Event(enable_timing=True)
        reps = max(1, min(steps, 3))
        a.record(stream)
        for _ in range(reps):
            for c, p in zip(ctxs, pss):
                c.step(p, dt=0.0, cfl=CFL, stream=stream)
        bb.record(stream)
        stream.synchronize()
        loop_ms = a.elapsed_time(bb) / reps
        for c in ctxs:
            c.close()
    return {"particles": n, "sims": nsim, "batched_ms": batched_ms, "loop_ms": loop_ms, "tune": tune,
            "launches": launches, "clocks": clocks, "steps": steps,
            "phases": {k: {"ms": v[0], "launches": v[1]} for k, v in phases.items() if v[1]}}


def run_ensemble(args):
    import torch
    torch.cuda.set_device(0)
    r = ensemble_measure(args, args.sims, args.steps, args.warmup)
    n, batched_ms, loop_ms = r["particles"], r["batched_ms"], r["loop_ms"]
    line = {"metric": METRIC, "value": n / (batched_ms * 1e-3), "unit": UNIT, "n_gpus": 1, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": batched_ms, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": "kh-ensemble-%d" % r["sims"], "particles": n, "dim": 2, "gamma": KH_GAMMA,
                       "sizes": "U[10k, 200k] per simulation (seed 6)", "schedule": "batched, CUDA graph replay",
                       "autotune": r["tune"], "l2": "flushed between timed steps (256 MiB write)"},
            "unbatched": {"ms_per_step": loop_ms, "value": n / (loop_ms * 1e-3),
                          "note": "one lp_step per simulation in a loop, one context each"},
            "speedup_vs_unbatched": loop_ms / batched_ms, "gpu_launches": r["launches"], "clocks": r["clocks"],
            "phases": r["phases"]}
    print(json.dumps(line), flush=True)


# ---------------------------------------------------------------------------
# the jet with reservoir inflow, grown to its end size
# ---------------------------------------------------------------------------

JET_H = 0.0169          # jet particle spacing: about 8M particles once the jet reaches z ~ 16


def run_inflow(args):
    """The jet grows from a short column above a Mach-3 reservoir inlet (1e3
    density contrast with the ambient): lp_step and lp_inflow each step, the
    arrays and the context's scratch doubled as the count grows (untimed).
    Once the count reaches the target, steps (lp_step + lp_inflow, the latter
    with its host read of the layer count) are timed."""
    import torch

    from paper_2206_11998_gb300 import build as b
    from paper_2206_11998_gb300 import inputs, lp

    b.build()
    torch.cuda.set_device(0)
    target = args.particles
    st, q = inputs.jet_inflow_3d(JET_H, density_ratio=args.density_ratio)
    n0 = st["V"].shape[0]
    inlet = lp.make_inlet(q["center"], q["axis"], q["radius"], q["spacing"], q["mass"], q["P_res"], q["rho_res"],
                          q["sample_depth"], ghost_layers=q["ghost_layers"], first_id=n0, ghost_id=2 ** 31)
    cap = 2 * n0
    cfg = lp.make_config(3, cap, kappa=KAPPA, k_max=K_MAX, k_side=8, gamma=inputs.JET_GAMMA, n_fluid=2 ** 31,
                         s_ref=(1.0, 1.0, 1.0, 3.5, 1.0),
                         limiter={"flagged": lp.LIM_FLAGGED, "uw": lp.LIM_UW}[args.limiter],
                         select={"nearest": lp.SELECT_NEAREST, "octant": lp.SELECT_OCTANT}[args.select])
    ctx = lp.Context(cfg)
    stream = torch.cuda.Stream()
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")
    growth = {"steps": 0, "reserves": 0}
    t0 = time.perf_counter()
    with torch.cuda.stream(stream):
        ps = lp.ParticleSet.with_capacity(st, cap)

        box_lo, box_hi = (-q["box"][0], -q["box"][0], -q["box"][1]), (q["box"][0], q["box"][0], q["box"][2])

        def advance():
            nonlocal ps
            ctx.step(ps, dt=0.0, cfl=CFL, stream=stream)
            growth["removed"] = growth.get("removed", 0) + ctx.remove_outside(ps, box_lo, box_hi, stream=stream)
            while True:
                try:
                    return ctx.inflow(ps, inlet, stream=stream)
                except lp.LPError as e:
                    if e.code != lp.ERR_CAPACITY:
                        raise
                    ps = ps.grown(2 * ps.capacity)
                    ctx.reserve(ps.capacity)
                    growth["reserves"] += 1

        ctx.inflow(ps, inlet, stream=stream)
        info = None
        tick = time.perf_counter()
        while ps.n < target and growth["steps"] < 4000 and time.perf_counter() - t0 < args.grow_seconds:
            info = advance()
            growth["steps"] += 1
            if growth["steps"] % 50 == 0:
                stream.synchronize()
                sg = ctx.stats(stream=stream)
                now = time.perf_counter()
                sys.stderr.write("grow step %d n %d dt %.3g  %.1f ms/step  layers %d  fp64-redo %d  query-fallback %d  "
                                 "rejected %d\n" % (growth["steps"], ps.n, sg["dt"], (now - tick) * 20.0,
                                                     info["layers_total"], sg["n_fp64_redo"], sg["n_query_fallback"],
                                                     sg["n_nonfinite"]))
                sys.stderr.flush()
                ctx.reset_stats(stream=stream)
                tick = now
        stream.synchronize()
        growth["reached_target"] = ps.n >= target
        growth["wall_s"] = time.perf_counter() - t0
        growth["start_particles"] = n0
        for _ in range(args.warmup):
            advance()
        ctx.reset_stats(stream=stream)
        ctx.phase_times(stream=stream)
        ctx.set_profiling(True)
        l0 = ctx.stats(stream=stream)["kernel_launches"]
        sampler = ClockSampler(gpu_index_for(0))
        sampler.start()
        ms, counts, infos = [], [], []
        for _ in range(args.steps):
            flush.zero_()
            a = torch.cuda.Event(enable_timing=True)
            e = torch.cuda.Event(enable_timing=True)
            counts.append(ps.n)
            a.record(stream)
            infos.append(advance())
            e.record(stream)
            e.synchronize()
            ms.append(a.elapsed_time(e))
        clocks = sampler.stop()
        ctx.set_profiling(False)
        phases = ctx.phase_times(stream=stream)
        s = ctx.stats(stream=stream)
    total_ms = sum(ms)
    value = sum(counts) / (total_ms * 1e-3)
    last = infos[-1]
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": 1, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": total_ms / args.steps, "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic",
            "config": {"workload": "jet-inflow-3d-%s" % size_tag(counts[0]), "particles_timed": [counts[0], ps.n],
                       "jet_spacing": JET_H, "inlet": {k: v for k, v in q.items() if k != "center"},
                       "limiter": args.limiter, "select": args.select,
                       "growth": growth, "flagged_per_step": s["n_flagged"] / args.steps,
                       "fp64_redo_per_step": s["n_fp64_redo"] / args.steps,
                       "rejected_updates_per_step": s["n_nonfinite"] / args.steps,
                       "l2": "flushed between timed steps (256 MiB write)"},
            "inflow": {"P_inf": last["P_inf"], "rho_inf": last["rho_inf"], "u_inf": last["u_inf"],
                       "mach": last["u_inf"] / last["c_inf"], "layers_per_step": sum(i["layers"] for i in infos) / len(infos),
                       "particles_per_layer": last["npat"]},
            "gpu_launches": s["kernel_launches"] - l0, "clocks": clocks,
            "phases": {k: {"ms_per_step": v[0] / args.steps, "launches": v[1]} for k, v in phases.items() if v[1]}}
    ctx.close()
    print(json.dumps(line), flush=True)


def estimator_compare(args):
    """The gas cloud advanced args.compare_estimators steps twice from the same
    state: with the plain estimator (CFL steps), and with the learned estimator
    trained on the cloud's own plain steps, taking the same sequence of steps so
    that both end at the same time.  Reports each run's time per step (CUDA
    events, eager steps), the flagged and skipped counts, and the learned run's
    drift from the plain one per field: the relative L2 and max differences of
    the final states, and the L2 difference relative to the plain run's own
    change from the initial state."""
    import torch

    from paper_2206_11998_gb300 import build as b
    from paper_2206_11998_gb300 import inputs, lp

    b.build()
    torch.cuda.set_device(0)
    steps = args.compare_estimators
    state = workload_state(args.particles)
    n = state["V"].shape[0]
    stream = torch.cuda.Stream()
    params, info = train_gate(lp, inputs, state, n, stream, torch)
    base = dict(radius_mode=lp.RADIUS_VOLUME, kappa=KAPPA, k_max=K_MAX, k_side=8, gamma=GAMMA,
                limiter=lp.LIM_FLAGGED, s_ref=inputs.field_scales(state))

    def run(ctx, dts):
        out_dt, ms, flagged, skipped, nonfinite = [], [], 0, 0, 0
        with torch.cuda.stream(stream):
            ps = lp.ParticleSet.from_state(state)
            ctx.reset_stats(stream=stream)
            for k in range(steps):
                e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                e0.record(stream)
                ctx.step(ps, dt=0.0 if dts is None else dts[k], cfl=CFL, stream=stream)
                e1.record(stream)
                if dts is None:
                    out_dt.append(ctx.stats(stream=stream)["dt"])
                ms.append((e0, e1))
            stream.synchronize()
            st = ctx.stats(stream=stream)
            idx = ps.id.long()
            byid = lambda t: torch.empty_like(t).index_copy_(0, idx, t)
            fields = {"V": byid(ps.V), "P": byid(ps.P)}
            for k in range(3):
                fields["u%d" % k] = byid(ps.u[k])
        t_ms = sum(a.elapsed_time(bb) for a, bb in ms) / steps
        return fields, out_dt, t_ms, st

    cp = lp.Context(lp.make_config(3, n, precision=lp.PREC_FP32, **base))
    fp, dts, ms_p, stp = run(cp, None)
    cp.close()
    cm = lp.Context(lp.make_config(3, n, precision=lp.PREC_FP32, estimator=lp.EST_MLP, mlp_tau_lo=info["tau_lo"],
                                   **base))
    cm.mlp_set_params(params)
    fm, _, ms_m, stm = run(cm, dts)
    cm.close()
    s0 = {"V": state["V"], "P": state["P"], "u0": state["u"][0], "u1": state["u"][1], "u2": state["u"][2]}
    drift = {}
    for nm in fp:
        a, bb = fm[nm].double(), fp[nm].double()
        z = torch.as_tensor(np.asarray(s0[nm]), device=a.device, dtype=torch.float64)
        d = a - bb
        drift[nm] = {"l2": float(d.norm() / max(float(bb.norm()), 1e-300)),
                     "max": float(d.abs().max() / max(float(bb.abs().max()), 1e-300)),
                     "l2_of_change": float(d.norm() / max(float((bb - z).norm()), 1e-300))}
    line = {"metric": "plain vs learned state estimator, %d steps" % steps, "impl": "ours",
            "config": config_dict(n, {"steps_compared": steps, "t_end": float(sum(dts)),
                                      "dt_first": dts[0], "dt_last": dts[-1]}),
            "plain": {"ms_per_step": ms_p, "value": n / (ms_p * 1e-3), "flagged_per_step": stp["n_flagged"] / steps,
                      "nonfinite": stp["n_nonfinite"], "fp64_redo_per_step": stp["n_fp64_redo"] / steps},
            "learned": {"ms_per_step": ms_m, "value": n / (ms_m * 1e-3),
                        "skipped_per_step": stm["n_mlp_skip"] / steps, "flagged_per_step": stm["n_flagged"] / steps,
                        "nonfinite": stm["n_nonfinite"], "gate": info},
            "drift_of_learned_from_plain": drift,
            "note": "eager lp_step calls timed with CUDA events (no L2 flush); the learned run takes the plain "
                    "run's CFL steps, so both states are at the same time"}
    return line


def main():
    args = parse()
    select_workload(args)
    if args.compare_estimators > 0 and args.impl != "reference":
        print(json.dumps(estimator_compare(args)), flush=True)
        return
    if args.impl == "reference":
        run_reference(args)
    elif args.workload == "kh-ensemble":
        run_ensemble(args)
    elif args.workload == "jet-inflow":
        run_inflow(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
