#!/usr/bin/env python
"""Benchmark of the hot path: multistep EPI steps of the DFR shallow-water
model on the rotated cubed sphere, with complex-step JVPs inside the adaptive
Krylov phi-function solver (arXiv 2101.05617, Sec. 3-4).

Workload (default): 6 x 60 x 60 elements, p = 5 (2,332,800 unknowns), EPI5,
dt = 1800 s, KIOPS tolerance 1e-10, seeded synthetic fields (degree <= 4
spherical-harmonic height around 8 km, geostrophic wind, seeded rotation).
A step = one EPI5 step (RHS, remainder JVPs, one KIOPS call with its JVPs,
orthogonalisation and exponentials, assembly).  The first P = 3 steps of the
run are EPI2 start-up steps and fall in the warm-up.

    python bench.py [--gpus N] [--steps K] [--warmup W] [--impl reference]

Prints one JSON line on rank 0.  Multi-GPU runs are independent replicas (one
per GPU, seed offset by rank): the path has no exchange step at one replica per
GPU; value = steps of all ranks / slowest rank's time.
"""
import argparse
import json
import os
import statistics
import subprocess
import sys
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "EPI steps/s and JVP DOF/s at n_e=60,p=5 vs plain FP64 GPU path, same error"
UNIT = "EPI steps/s"


def flops_per_jvp(ne, ns, p=4, dots=True):
    """Algorithmic FP64 flops of one Krylov JVP of the split path (the imaginary
    half of the complex-step evaluation at a fixed linearisation point; add /
    mul = 1, fma = 2) with the augmented-operator epilogue of p phi-vectors and
    the two dot products of the new vector with the window (not the window's own
    product, which the kernel forms beside them), split into the volume and face
    kernels.  Most of them run as integer operations (block fixed point), so
    their rate is no fraction of the FP64 peak.  Per node: pointwise imaginary fluxes and sources 23, DFR sweeps
    27 + 12 Ns, scaling 3, epilogue 7 p (+ 12 with the dots).  Per interface
    point: traces 12 Ns, the 3 x 6 flux map 33, hand-back 7."""
    nodes = 6 * ne * ne * ns * ns
    facepts = 12 * ne * ne * ns
    vol = 23 + 27 + 12 * ns + 3 + 7 * p + (12 if dots else 0)
    return nodes * vol, facepts * (12 * ns + 40)


# DRAM bytes (read + write) of one launch of the dominant kernel,
# volume_tangent_kernel<double, 6>, on the 6 x 60 x 60, p = 5 workload inside
# the phi-function solver (p = 4, with dots), from one ncu capture of the
# kernel as it stands (dram__bytes_read.sum + dram__bytes_write.sum); none
# while the kernel has changed since its last capture.
TRAFFIC_BYTES = {"ne60_p5": 188.05e6}   # 176.23 MB read + 11.83 MB written

# phi-vectors phi_1 .. phi_M of an EPI order (the b columns of its phi-function call)
EPI_PHI = {2: 1, 3: 2, 4: 3, 5: 4, 6: 4}

# the timed region brackets every PROFILE_EVERY-th launch of the dominant kernel
# with CUDA events (its average launch duration for the roofline)
PROFILE_EVERY = 16


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=12)
    ap.add_argument("--warmup", type=int, default=4)
    ap.add_argument("--impl", default="gpu", choices=["gpu", "reference"])
    ap.add_argument("--workload", default="ne60_p5")
    ap.add_argument("--seed", type=int, default=0)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-forms", action="store_true")
    ap.add_argument("--no-ensemble", action="store_true")
    ap.add_argument("--no-large", action="store_true",
                    help="skip the 6x90x90, p=6 EPI6 instance (FP64 and complex64-bulk, per-kernel rooflines)")
    ap.add_argument("--only-forms", default="",
                    help="comma-separated forms to run (learned, ne30, ne60, ensemble, large); default all")
    ap.add_argument("--control", default="plain", choices=["learned", "plain"])
    ap.add_argument("--oracle-full-step", action="store_true",
                    help="time one complete oracle EPI step of the workload on one host core and exit")
    ap.add_argument("--jvp-mode", type=int, default=1, choices=[0, 1, 2],
                    help="0: full complex-step evaluation per JVP, 1: split (default), 2: complex64-bulk "
                         "(--kiops-call only; the timed step is the FP64 path)")
    ap.add_argument("--kiops-call", action="store_true",
                    help="one phi-function call on the workload (b = [0, dt F, 1e-3 dt F shifted, ...]) with "
                         "--jvp-mode, --iop and --m-max, then exit: the small case for kernel profiles")
    ap.add_argument("--iop", type=int, default=2)
    ap.add_argument("--m-max", type=int, default=24)
    return ap.parse_args()


def dist_setup(args):
    world = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    pg = None
    if world > 1:
        import torch
        import torch.distributed as dist
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        backend = "nccl" if torch.cuda.is_available() and args.impl == "gpu" else "gloo"
        if backend == "nccl":
            torch.cuda.set_device(local)
        # rank 0 alone runs the one-rank extras while the others wait at the final barrier
        import datetime
        dist.init_process_group(backend, timeout=datetime.timedelta(minutes=30))
        pg = dist
    return world, rank, local, pg


def aggregate(pg, elapsed_ms, steps, device=None):
    """(max elapsed over ranks, total steps over ranks): value = total / max."""
    if pg is None:
        return elapsed_ms, steps
    import torch
    t = torch.tensor([elapsed_ms], dtype=torch.float64, device=device)
    s = torch.tensor([float(steps)], dtype=torch.float64, device=device)
    pg.all_reduce(t, op=pg.ReduceOp.MAX)
    pg.all_reduce(s, op=pg.ReduceOp.SUM)
    return float(t.item()), int(s.item())


class ClockSampler:
    """nvidia-smi clock/throttle samples during the timed region."""
    Q = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index):
        self.proc = None
        self.gpu = gpu_index

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.Q}", "--format=csv,noheader,nounits",
                                          "-lms", "200", "-i", str(self.gpu)], stdout=subprocess.PIPE,
                                         stderr=subprocess.DEVNULL, text=True)
        except (OSError, FileNotFoundError):
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
            parts = [p.strip() for p in line.split(",")]
            if len(parts) < 7:
                continue
            try:
                sm.append(float(parts[0]))
                smax.append(float(parts[1]))
            except ValueError:
                continue
            for nm, val in zip(names, parts[3:7]):
                if val.lower() == "active":
                    reasons.add(nm)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


class _SampleDone(Exception):
    pass


def oracle_setup(wl, seed):
    """The oracle's grid, state and phi-vectors of an EPI step of the workload
    (not timed)."""
    import numpy as np

    from oracle import fields as ofields
    from oracle import shallow_water as osw
    from paper_2101_05617_gb300 import synth
    f = synth.make_fields(wl, seed)
    g = osw.Grid(wl.ne, wl.ns, f.rotation)
    h, hB, V = f.evaluate(g.node_xyz())
    q = ofields.state_from_fields(g, h, hB, V)
    v = synth.random_perturbation(q.size, seed + 1).reshape(q.shape)
    F = osw.rhs_real(g, q).reshape(-1)
    M = {2: 1, 3: 2, 4: 3, 5: 4, 6: 4}[wl.order]
    b = [np.zeros(q.size), wl.dt * F] + [1e-3 * wl.dt * np.roll(F, 7 * k + 1) for k in range(M - 1)]
    return {"g": g, "q": q, "v": v, "b": b, "dt": wl.dt, "tol": wl.tol, "seed": seed}


def oracle_kiops_sample(st, budget_s=15.0):
    """Time the oracle, as it stands, on a bounded sample of the workload at full
    size (state from oracle_setup): its RHS, one standalone complex-step JVP,
    its KIOPS (the augmented JVP plus the incomplete orthogonalisation of every
    Krylov iteration; Krylov size 128 from the first iteration) on the
    phi-vectors of an EPI step until ~budget_s have passed, scipy's expm of a
    (129 x 129) augmented Hessenberg matrix (the oracle's exponential) and a
    basis combination.  Returns the per-unit costs in seconds."""
    import numpy as np
    import scipy.linalg

    from oracle import kiops as okiops
    from oracle import shallow_water as osw
    g, q, v, dt = st["g"], st["q"], st["v"], st["dt"]
    t0 = time.perf_counter()
    osw.rhs_real(g, q)
    t_rhs = time.perf_counter() - t0
    t0 = time.perf_counter()
    osw.jvp(g, q, v)
    t_jvp = time.perf_counter() - t0
    calls = [0]
    tk = [time.perf_counter()]

    def matvec(x):
        if calls[0] >= 2 and time.perf_counter() - tk[0] > budget_s:
            raise _SampleDone()
        calls[0] += 1
        return dt * osw.jvp(g, q, x.reshape(q.shape)).reshape(-1)
    tk[0] = time.perf_counter()
    try:
        okiops.kiops(1.0, matvec, st["b"], tol=st["tol"], m_init=128, m_min=10, m_max=128)
    except _SampleDone:
        pass
    t_iter = (time.perf_counter() - tk[0]) / max(1, calls[0])
    rng = np.random.default_rng(st["seed"])
    Hm = np.triu(rng.standard_normal((129, 129)), -1) * 0.05
    Hm[0, 128] = 1.0
    t0 = time.perf_counter()
    scipy.linalg.expm(Hm)
    t_expm = time.perf_counter() - t0
    Vs = rng.standard_normal((16, q.size))
    c = rng.standard_normal(16)
    t0 = time.perf_counter()
    _ = Vs.T @ c
    t_comb16 = time.perf_counter() - t0
    return {"t_rhs": t_rhs, "t_jvp": t_jvp, "t_iter": t_iter, "iters": calls[0], "t_expm": t_expm,
            "t_combine_128": t_comb16 * 8.0}


def project_oracle_step(s, krylov, attempts, substeps, P):
    """EPI step time of the oracle composed from its measured per-unit costs and a
    step's counts: Krylov iterations, substep attempts (one exponential each),
    accepted substeps (one combination each), P remainder JVPs and one RHS."""
    return (krylov * s["t_iter"] + attempts * s["t_expm"] + substeps * s["t_combine_128"] + P * s["t_jvp"]
            + s["t_rhs"])


def oracle_sample(wl, seed, counts, P, budget_s=15.0):
    """cpu_baseline: the oracle's step time on one host core, PROJECTED from a
    bounded sample (oracle_kiops_sample) with the Krylov iterations, substep
    attempts and accepted substeps per step that this run measured (the
    oracle's KIOPS takes the same decisions: the parity tests check identical
    counts)."""
    s = oracle_kiops_sample(oracle_setup(wl, seed), budget_s)
    k, a, sub = counts
    step_s = project_oracle_step(s, k, a, sub, P)
    return {"value": 1.0 / step_s, "unit": UNIT, "cores": 1, "kind": "oracle", "projected": True,
            "sample": (f"oracle KIOPS at n_e={wl.ne}, p={wl.p} (full size): {s['iters']} Krylov iterations "
                       f"(augmented JVP + incomplete orthogonalisation) in {s['iters'] * s['t_iter']:.1f} s, "
                       f"1 RHS, 1 JVP, 1 scipy expm (129x129), 1 basis combination; EPI{wl.order} step PROJECTED "
                       f"with this run's mean counts per step: {k:.0f} Krylov iterations, {a:.1f} substep attempts, "
                       f"{sub:.1f} accepted substeps, {P} remainder JVPs, 1 RHS"),
            "per_unit_s": {"krylov_iteration": s["t_iter"], "jvp": s["t_jvp"], "rhs": s["t_rhs"],
                           "expm_129": s["t_expm"], "combine_128": s["t_combine_128"]},
            "jvp_dof_per_s": wl.n_unknowns / s["t_jvp"]}


def _oracle_jvp_worker(args):
    """One host process of the all-cores oracle sample: build the oracle grid,
    meet the other workers, then time complex-step JVPs for budget_s."""
    wl_name, seed, budget_s = args
    from oracle import fields as ofields
    from oracle import shallow_water as osw
    from paper_2101_05617_gb300 import synth
    wl = synth.WORKLOADS[wl_name]
    f = synth.make_fields(wl, seed)
    g = osw.Grid(wl.ne, wl.ns, f.rotation)
    h, hB, V = f.evaluate(g.node_xyz())
    q = ofields.state_from_fields(g, h, hB, V)
    v = synth.random_perturbation(q.size, seed + 1).reshape(q.shape)
    _worker_barrier.wait(timeout=600)
    t0 = time.perf_counter()
    n = 0
    while time.perf_counter() - t0 < budget_s or n < 1:
        osw.jvp(g, q, v)
        n += 1
    return n, time.perf_counter() - t0


_worker_barrier = None


def _oracle_pool_init(barrier):
    global _worker_barrier
    _worker_barrier = barrier


def oracle_sample_all_cores(wl, seed, krylov_per_step, P, single, budget_s=15.0):
    """The same oracle sample on every host core: one unchanged oracle process
    per core computing JVPs of the full-size workload concurrently (started
    together); the step is projected from the aggregate JVP rate as for the
    one-core sample (RHS and orthogonalisation terms taken from it)."""
    import multiprocessing as mp
    k = max(1, min(16, os.cpu_count() or 1))
    ctx = mp.get_context("spawn")
    barrier = ctx.Barrier(k)
    try:
        with ctx.Pool(k, initializer=_oracle_pool_init, initargs=(barrier,)) as pool:
            res = pool.map_async(_oracle_jvp_worker, [(wl.name, seed, budget_s)] * k,
                                 chunksize=1).get(timeout=budget_s + 900)
    except Exception as e:   # a worker that died or timed out: report, do not block the benchmark
        return {"unavailable": f"{type(e).__name__}: {e}"[:200], "cores": k, "kind": "oracle"}
    rate = sum(n / t for n, t in res)             # JVPs per second, all processes
    t_one = 1.0 / rate
    step_s = 1.0 / single["value"]
    jvp_single = single["per_unit_s"]["jvp"]
    step_s = step_s - (krylov_per_step + P) * jvp_single + (krylov_per_step + P) * t_one
    return {"value": 1.0 / step_s, "unit": UNIT, "cores": k, "kind": "oracle", "projected": True,
            "sample": (f"{sum(n for n, _ in res)} oracle complex-step JVPs in {k} concurrent processes "
                       f"(~{budget_s:.0f} s each) at n_e={wl.ne}, p={wl.p}; EPI{wl.order} step PROJECTED: the "
                       f"one-core projection with its JVP time replaced by the aggregate JVP rate (the "
                       f"orthogonalisation, expm and combination terms stay single-core)"),
            "jvp_dof_per_s": wl.n_unknowns * rate}


def hbm_peak_gbs():
    """The measured HBM copy bandwidth of the GB300s (GB/s), else the fallback."""
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as fh:
            return float(json.load(fh)["hbm_gbs"]), "measured"
    except (OSError, KeyError, ValueError):
        return 6800.0, "fallback"


def ortho_roofline(prof_all, wl, fused):
    """The two vector passes of the window-2 orthogonalisation in one launch
    (fused; else not reported) against HBM: algorithmic bytes per Krylov iteration
    (orth_bytes_per_unknown) per unknown of the augmented vector; the fused launch
    counts as the two passes."""
    o = prof_all["orthogonalisation"]
    if not o["count"] or not fused:
        return None
    pairs = o["count"] / 2.0
    t = o["ms"] * 1e-3 / pairs
    nbytes = orth_bytes_per_unknown(2, 1, True) * (wl.n_unknowns + 4)
    peak, src = hbm_peak_gbs()
    return {"bound": "hbm", "bytes_per_iteration": nbytes, "avg_ms_per_iteration": t * 1e3,
            "achieved_gbs": nbytes / t / 1e9, "peak_gbs": peak, "frac": nbytes / t / 1e9 / peak,
            "peak_source": src}


def volume_bytes_per_node(ns, mode, iop, p):
    """Bytes one volume-kernel launch of a Krylov iteration must move per node:
    read v (3 doubles; its FP32 copy in the complex64-bulk form) and write Jv (3
    doubles), read the iop orthogonalisation window vectors (3 iop doubles; none in
    the complex64-bulk form, whose dots are a pass of their own), the p
    b-column vectors of the augmented operator (3 p entries: FP64, or their FP32
    copies in the complex64-bulk form), the 11 split-JVP coefficients (FP64, or
    FP32 in the complex64-bulk form) and the interface fluxes of the element's four
    edges (12 N_s values per element = 12 / N_s per node, FP64 or FP32)."""
    w = 8 if mode == 1 else 4
    window = 24 * iop if mode == 1 else 0   # the complex64-bulk form's volume kernel reads no window vectors
    return 3 * w + 24 + window + 3 * p * w + 11 * w + 12.0 / ns * w


def face_bytes_per_node(ns, mode=1):
    """Bytes the face kernel of a Krylov iteration must move per node: v read once
    (its FP32 copy in the complex64-bulk form), per interface point the 18 flux-map
    coefficients and the three fluxes handed to both sides (12 n_e^2 N_s points, 2 /
    N_s per node; FP64, or FP32 in the complex64-bulk form)."""
    w = 8 if mode == 1 else 4
    return 3 * w + (18 + 2 * 3) * w * 2.0 / ns


def full_bytes_per_node(ns, kernel, iop, p):
    """The same for the full complex-step evaluation (--jvp-mode 0): the face
    kernel reads q and v, per interface point 12 coefficients, and hands over three
    fluxes twice; the volume kernel reads q, v, 13 coefficients, the interface
    fluxes, the window and the b-columns and writes Jv."""
    if kernel == "face":
        return 48 + (12 * 8 + 2 * 3 * 8) * 2.0 / ns
    return 48 + 24 + 13 * 8 + 12.0 / ns * 8 + 24 * iop + 24 * p


def orth_bytes_per_unknown(iop, mode=1, fused=False):
    """The vector passes of the window-iop orthogonalisation per unknown of the
    augmented vector.  In one launch (fused, what the benchmark times and
    reports): each vector once, read z and the window vectors, write V_{j+1} = 8
    (iop + 2) B; in the complex64-bulk form the launch also forms the window dots
    and writes the FP32 copy: 8 (iop + 2) + 4 B.  Not fused: the count of a
    second pass that reads iop - 1 window vectors for the next dots, 8 (2 iop + 3)
    B, in the complex64-bulk form 8 (iop + 2) + 20 B; the library's second launch
    forms no dots any more (8 (iop + 4) B for the two), and the benchmark does not
    report that form."""
    if fused:
        return 8.0 * (iop + 2) + (4.0 if mode == 2 else 0.0)
    if mode == 2:
        return 8.0 * (iop + 2) + 20.0
    return 8.0 * (2 * iop + 3)


def kernel_rooflines(prof, wl, mode, iop, step_ms, fp64_peak=None, fused=False):
    """Per-kernel figures of one EPI step with every kernel family bracketed by
    events: the algorithmic bytes (volume_bytes_per_node, face_bytes_per_node,
    orth_bytes_per_unknown) against the measured copy bandwidth, and the rate of
    the algorithmic flops (flops_per_jvp, 6 more per node for the third dot of
    window 3).  fp64_peak: for kernels that run those flops on the FP64 pipe, also
    their fraction of it (the library's split kernels do not, see flops_per_jvp)."""
    hbm, _ = hbm_peak_gbs()
    nodes = 6 * wl.ne * wl.ne * wl.ns * wl.ns
    p = EPI_PHI[wl.order]
    fv, ff = flops_per_jvp(wl.ne, wl.ns)
    fv += 6 * nodes * (iop - 2)
    out = {}

    def avg(kind):
        k = prof[kind]
        return k["ms"] / k["count"] * 1e-3 if k["count"] else None
    tv, tf, to = avg("volume_jvp"), avg("face_jvp"), avg("orthogonalisation")
    if tv:
        vbytes = nodes * volume_bytes_per_node(wl.ns, mode, iop, p)
        v = {"avg_us": tv * 1e6, "launches": prof["volume_jvp"]["count"], "flops": fv,
             "bytes": vbytes, "gbs": vbytes / tv / 1e9, "hbm_frac": vbytes / tv / 1e9 / hbm}
        if mode == 1:
            v["tflops"] = fv / tv / 1e12
            if fp64_peak:
                v["fp64_frac"] = v["tflops"] / fp64_peak
        else:
            v["fp32_tflops"] = fv / tv / 1e12
        out["volume"] = v
    if tf:
        fbytes = nodes * face_bytes_per_node(wl.ns, mode)
        f = {"avg_us": tf * 1e6, "launches": prof["face_jvp"]["count"], "flops": ff,
             "bytes": fbytes, "gbs": fbytes / tf / 1e9, "hbm_frac": fbytes / tf / 1e9 / hbm}
        f["tflops" if mode == 1 else "fp32_tflops"] = ff / tf / 1e12
        out["face"] = f
    if to:
        t = 2.0 * to   # the update and the scaling of a Krylov iteration count as two passes, in one launch or two
        obytes = orth_bytes_per_unknown(iop, mode, fused) * (wl.n_unknowns + 4)
        out["orthogonalisation"] = {"avg_us_per_iteration": t * 1e6, "bytes_per_iteration": obytes,
                                    "gbs": obytes / t / 1e9, "hbm_frac": obytes / t / 1e9 / hbm}
    if prof["expm"]["count"]:
        out["expm"] = {"avg_us": avg("expm") * 1e6, "launches": prof["expm"]["count"]}
    out["share_of_step"] = {k: prof[k]["ms"] / step_ms
                            for k in ("volume_jvp", "face_jvp", "orthogonalisation", "expm", "linearize")}
    out["peaks"] = {"hbm_gbs": hbm}
    return out


def fp32_form_comparison(args, dev, workload="ne30_p5", variants=(("fp64", 1, 2), ("complex64_bulk", 2, 2)),
                         per_kernel=False, total_steps=None, dt=None):
    """The complex64-bulk form against the FP64 path: steps/s of each variant
    (name, JVP mode, orthogonalisation window[, "learned": the learned initial
    substep after the warm-up]) from the same start, each variant's state
    difference to the first (the FP64 path, window 2) after the run, and the EPI
    time-discretisation error (FP64 at dt against dt/4).  With per_kernel, each
    variant then takes one more step with every kernel family bracketed by
    events (after its state was kept) and reports per-kernel rooflines."""
    import torch

    from paper_2101_05617_gb300 import learned, swepi, synth
    wl = synth.WORKLOADS[workload]
    f = synth.make_fields(wl, args.seed)
    warm = args.warmup
    timed = args.steps if total_steps is None else total_steps - warm
    res = {}
    states = {}
    kernels = {}
    stats = {}
    dt0 = wl.dt if dt is None else dt
    runs = [(v[0], v[1], v[2], dt0, 1, v[3] if len(v) > 3 else "") for v in variants]
    runs.append(("fp64_dt4", 1, 2, dt0 / 4, 4, ""))
    ctl = None
    fields = None   # the same grid and rotation for every run: evaluate the fields once
    for name, mode, iop, dt, mult, extra in runs:
        use_ctl = extra == "learned"
        ctx = swepi.SWContext(wl.ne, wl.p, f.rotation)
        if fields is None:
            fields = f.evaluate(ctx.node_xyz())
        q = torch.tensor(ctx.state_from_fields(*fields), device=dev)
        ctx.set_jvp_mode(mode)
        if extra == "device":   # the phi-function solver's controller on the device (one CUDA graph per call)
            ctx.set_kiops_driver(1)
        # both vector passes in one launch (the device controller's graph keeps two, but a profiled step runs the
        # host controller)
        fused = bool(ctx.set_orth_fused(1))
        h0max = float(q.view(3, -1)[0].abs().max())
        done = 0   # EPI steps completed (reported with a failure)
        try:
            for _ in range(warm * mult):
                ctx.epi_step(wl.order, dt, q, tol=wl.tol, iop=iop)
                done += 1
            if use_ctl:
                ctl = ctl or learned.Controller.load()
                swepi.sw_set_controller(ctx.handle, ctl.handle)
            torch.cuda.synchronize()
            e0 = torch.cuda.Event(enable_timing=True)
            e1 = torch.cuda.Event(enable_timing=True)
            kry = 0
            e0.record()
            for _ in range(timed * mult):
                kry += ctx.epi_step(wl.order, dt, q, tol=wl.tol, iop=iop)["krylov_iters"]
                done += 1
            e1.record()
            torch.cuda.synchronize()
            res[name] = timed * mult / (e0.elapsed_time(e1) * 1e-3)
            stats[name] = kry / (timed * mult)
            states[name] = q.view(3, -1).clone()
            if per_kernel and mult == 1:
                try:   # a failure here leaves the variant's timing and state in place
                    ctx.profile(True)
                    b0 = torch.cuda.Event(enable_timing=True)
                    b1 = torch.cuda.Event(enable_timing=True)
                    b0.record()
                    ctx.epi_step(wl.order, dt, q, tol=wl.tol, iop=iop)
                    b1.record()
                    torch.cuda.synchronize()
                    kernels[name] = kernel_rooflines(ctx.profile_read(), wl, mode, iop, b0.elapsed_time(b1),
                                                     fused=fused)
                    if not fused:
                        kernels[name].pop("orthogonalisation", None)
                except Exception as e:
                    kernels[name] = {"error": f"{type(e).__name__}: {e}"[:200]}
                ctx.profile(False)
        except Exception as e:   # e.g. a variant that left the finite range: reported per variant
            torch.cuda.synchronize()
            growth = float(q.view(3, -1)[0].abs().max()) / h0max
            res[name] = (f"{type(e).__name__}: {e}"[:160] + f" in step {done + 1}; max |q^0| at the failing "
                         f"step's start / initial = {growth:.3g}")
            states[name] = None
        swepi.sw_set_controller(ctx.handle, None)
        ctx.close()

    def rel(a, b):
        return [float(torch.linalg.norm(a[k] - b[k]) / torch.linalg.norm(b[k])) for k in range(3)]
    base = variants[0][0]
    ok = lambda k: states.get(k) is not None   # noqa: E731
    out = {"workload": f"{workload}: 6x{wl.ne}x{wl.ne} elements, p={wl.p}, EPI{wl.order}, dt={dt0:g} s, "
                       f"KIOPS tol {wl.tol:g}",
           "steps": warm + timed, "timed_steps": timed,
           "time_discretisation_err_rel_l2": rel(states[base], states["fp64_dt4"])
           if ok(base) and ok("fp64_dt4") else None}
    for v in variants:
        name, mode, iop = v[0], v[1], v[2]
        out[name] = {"jvp": "FP64" if mode == 1 else "complex64 bulk (FP32 imaginary half)", "window": iop,
                     "control": "learned" if len(v) > 3 and v[3] == "learned" else "plain",
                     "controller_on": "device" if len(v) > 3 and v[3] == "device" else "host"}
        if not ok(name):
            out[name]["error"] = res[name]
            continue
        out[name]["steps_per_s"] = res[name]
        out[name]["krylov_iters_per_step"] = stats.get(name)
        out[name]["finite"] = bool(torch.isfinite(states[name]).all())
        if ok(base):
            out[name]["speedup_vs_" + base] = res[name] / res[base]
            if name != base:
                out[name]["err_vs_" + base + "_rel_l2"] = rel(states[name], states[base])
        if name in kernels:
            out[name]["kernels"] = kernels[name]
    return out


# The largest time step (of 1200, 900, 600 s) at which EPI6 on the 6 x 90 x 90,
# p = 6 workload stays stable over its 36 steps on the GB300 (FP64 path,
# diagnostics after every step; the complex64-bulk form behaves the same).
LARGE_STABLE_DT = 600.0

# One complete oracle EPI5 multistep step on the default workload (6 x 60 x 60,
# p = 5; history q_{n-i} = q_n - i dt F(q_n)), measured on one host core by
# `python bench.py --oracle-full-step`: its own KIOPS counts (used to project the
# reference arm's sampled step) and its wall time.
ORACLE_STEP_NE60_P5 = {"krylov_iters": 384, "attempts": 13, "substeps": 3, "seconds": 342.3,
                       "host": "one x86-64 core of the build container (the counts do not depend on the host)"}


def ensemble_form(args, dev):
    """The batched ensemble: 96 members on uneven grids (n_e in {8, 16, 24, 32},
    p in {3, 4, 5}, EPI4/5, dt = 900 s, degree <= 12 perturbations of 50 m)
    for 24 steps through sw_ens_epi_run after autotuning; against one member
    per (n_e, p) class run alone through sw_epi_step (rate and state difference)."""
    import torch
    from paper_2101_05617_gb300 import ensemble, swepi, synth
    members = synth.ensemble_members(96, seed=args.seed)
    steps = 24
    t0 = time.perf_counter()
    ctxs, qs = ensemble.build(members)
    build_s = time.perf_counter() - t0
    ens = swepi.SWEnsemble(ctxs)
    block = ens.tune(qs, iters=4)
    tiles = {}
    for i, m in enumerate(members):
        tiles[f"ne{m.ne}_p{m.p}"] = ens.tiles(i)
    orders = [m.order for m in members]
    dts = [m.dt for m in members]
    ys = [q.clone() for q in qs]
    ens.epi_run(1, orders, dts, ys, tol=1e-10)                 # warm-up: first-touch allocations
    ensemble.reset(ctxs)
    ys = [q.clone() for q in qs]
    ens.profile(True)
    torch.cuda.synchronize()
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    e0.record()
    st = ens.epi_run(steps, orders, dts, ys, tol=1e-10)
    e1.record()
    torch.cuda.synchronize()
    sec = e0.elapsed_time(e1) * 1e-3
    info = ens.stats()
    ens.close()
    krylov = [a["krylov_iters"] for a in st]
    # one member per class alone, same start, same steps
    pick = {}
    for i, m in enumerate(members):
        pick.setdefault((m.ne, m.p), i)
    idx = sorted(pick.values())
    refs, ref_st, single_s = ensemble.run_single([members[i] for i in idx], [ctxs[i] for i in idx],
                                                 [qs[i] for i in idx], steps, tol=1e-10)
    same_krylov = sum(int(st[i]["krylov_iters"] == r["krylov_iters"]) for i, r in zip(idx, ref_st))
    diff = 0.0
    for i, r in zip(idx, refs):
        a, b = ys[i].view(3, -1), r.view(3, -1)
        diff = max(diff, max(float(torch.linalg.norm(a[k] - b[k]) / torch.linalg.norm(b[k])) for k in range(3)))
    fl = nb = 0.0
    for m, k in zip(members, krylov):
        fl += k * sum(flops_per_jvp(m.ne, m.ns, p=m.order - 1))
        # the update task reads z and two window vectors and writes z, the scaling reads and writes it: 48 B
        nb += k * m.nodes * (volume_bytes_per_node(m.ns, 1, 2, EPI_PHI[m.order]) + face_bytes_per_node(m.ns) + 3 * 48)
    iter_s = info["iter_ms"] * 1e-3
    hbm, _ = hbm_peak_gbs()
    return {"members": len(members), "steps": steps, "seconds": sec,
            "members_per_s": len(members) / sec, "member_steps_per_s": len(members) * steps / sec,
            "jvp_dof_per_s": sum(k * 3 * m.nodes for m, k in zip(members, krylov)) / sec,
            "unknowns_total": sum(3 * m.nodes for m in members),
            "krylov_iters": {"total": sum(krylov), "max_member": max(krylov)},
            "batched_iterations": info["ticks"], "read_backs": info["reads"], "expm_batches": info["expm_batches"],
            "gpu_launches": info["launches"], "block": info["block"], "ctas": info["ctas"],
            "tiles_by_class": tiles,
            "iteration_kernel": {"ms": info["iter_ms"], "share_of_run": info["iter_ms"] * 1e-3 / sec,
                                 "tflops": fl / iter_s / 1e12 if iter_s > 0 else None, "bytes": nb,
                                 "gbs": nb / iter_s / 1e9 if iter_s > 0 else None,
                                 "hbm_frac": nb / iter_s / 1e9 / hbm if iter_s > 0 else None},
            "single_member_path": {"members": len(idx), "seconds": single_s,
                                   "member_steps_per_s": len(idx) * steps / single_s},
            "max_rel_l2_vs_single": diff, "members_with_equal_krylov_count": same_krylov, "build_s": build_s}


def headline(out):
    """The metric's own comparison in a few keys (kept last on the line): the
    learned + complex64-bulk form against the plain FP64 GPU path on the same
    grid and start, with both errors against the FP64 path: the form's, and the
    EPI time-discretisation error (FP64 at dt against dt/4)."""
    c = out.get("forms", {}).get("complex64_bulk_ne60_p5")
    h = {"fp64_steps_per_s": out["value"], "fp64_e2e_steps_per_s": out["e2e"]["value"]}
    if not isinstance(c, dict) or "fp64" not in c:
        return h
    base = c["fp64"].get("steps_per_s")
    td = c.get("time_discretisation_err_rel_l2")
    h.update({"steps": c.get("steps"), "fp64_same_start_steps_per_s": base,
              "time_disc_err": max(td) if td else None})
    for key, name in (("learned_c64", "complex64_bulk_window3_learned"), ("plain_c64", "complex64_bulk_window3")):
        v = c.get(name, {})
        if "steps_per_s" in v:
            e = v.get("err_vs_fp64_rel_l2")
            h[key] = {"steps_per_s": v["steps_per_s"], "speedup": v.get("speedup_vs_fp64"),
                      "err_vs_fp64": max(e) if e else None, "finite": v.get("finite")}
        else:
            h[key] = {"error": str(v.get("error", "not run"))[:80]}
    return h


def run_reference(args, world, rank):
    """The oracle arm: each step times a bounded sample of the oracle on the full
    workload (oracle_kiops_sample, ~2 s of KIOPS iterations plus its RHS, JVP,
    expm and combination) and PROJECTS the EPI step from it with the oracle's
    own KIOPS counts of one complete measured step (ORACLE_STEP_NE60_P5)."""
    from paper_2101_05617_gb300 import synth
    if rank != 0:
        return
    wl = synth.WORKLOADS[args.workload]
    P = {2: 0, 3: 1, 4: 2, 5: 3, 6: 4}[wl.order]
    ref = ORACLE_STEP_NE60_P5
    counts = (ref["krylov_iters"], ref["attempts"], ref["substeps"])
    st = oracle_setup(wl, args.seed)
    times, sampled = [], 0.0
    t_all = time.perf_counter()
    for k in range(args.warmup + args.steps):
        t0 = time.perf_counter()
        s = oracle_kiops_sample(st, budget_s=2.0)
        if k >= args.warmup:
            times.append(project_oracle_step(s, *counts, P))
            sampled += time.perf_counter() - t0
    step_s = statistics.mean(times)
    value = 1.0 / step_s
    sample = (f"per step: the oracle's KIOPS at n_e={wl.ne}, p={wl.p} (full size) for ~2 s of Krylov iterations, "
              f"1 RHS, 1 JVP, 1 scipy expm (129x129), 1 basis combination; the EPI{wl.order} step is PROJECTED with "
              f"the oracle's counts of one complete step ({counts[0]} Krylov iterations, {counts[1]} substep "
              f"attempts, {counts[2]} substeps, {P} remainder JVPs, 1 RHS)")
    out = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": args.gpus,
           "steps": args.steps, "warmup": args.warmup, "ms_per_step": step_s * 1e3, "higher_is_better": True,
           "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
           "config": {"workload": f"{wl.name}: 6x{wl.ne}x{wl.ne} elements, p={wl.p}, EPI{wl.order}, "
                                  f"dt={wl.dt:g} s, KIOPS tol {wl.tol:g}", "parallelism": "replicas"},
           "projected": True,
           "projection": {"sampled_seconds_timed": sampled, "run_seconds": time.perf_counter() - t_all,
                          "projected_seconds_timed": step_s * args.steps,
                          "oracle_complete_step": ref},
           "cpu_baseline": {"value": value, "unit": UNIT, "cores": 1, "kind": "oracle", "projected": True,
                            "sample": sample},
           "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(out), flush=True)


def run_kiops_call(args):
    """One phi-function call (Eq. 29) at the workload's first state: b_0 = 0,
    b_1 = dt F(q), b_2, b_3 = 1e-3 and 1e-4 dt F(q) shifted by 7 and 11 entries;
    Krylov size fixed at --m-max (tolerance 1e-6), window --iop, JVP form
    --jvp-mode.  Prints the solver statistics."""
    import torch

    from paper_2101_05617_gb300 import synth
    from paper_2101_05617_gb300.swepi import SWContext
    wl = synth.WORKLOADS[args.workload]
    f = synth.make_fields(wl, args.seed)
    ctx = SWContext(wl.ne, wl.p, f.rotation)
    q = torch.tensor(ctx.state_from_fields(*f.evaluate(ctx.node_xyz())), device="cuda")
    ctx.set_jvp_mode(args.jvp_mode)
    b1 = wl.dt * ctx.rhs(q)
    t0 = time.perf_counter()
    _, st = ctx.kiops_phi(q, wl.dt, [None, b1, 1e-3 * b1.roll(7), 1e-4 * b1.roll(11)], m_max=args.m_max, m_min=10,
                          m_init=args.m_max, iop=args.iop, tol=1e-6)
    torch.cuda.synchronize()
    print(json.dumps({"kiops_call": {"workload": wl.name, "jvp_mode": args.jvp_mode, "iop": args.iop,
                                     "m_max": args.m_max, "seconds": time.perf_counter() - t0, **st}}), flush=True)


def run_oracle_full_step(args):
    """One complete oracle EPI step of the workload on one host core, measured
    (not projected): history q_{n-i} = q_n - i dt F(q_n) for the P previous
    states, then the multistep step (RHS, remainder JVPs, one KIOPS call)."""
    import numpy as np

    from oracle import epi as oepi
    from oracle import shallow_water as osw
    from paper_2101_05617_gb300 import synth
    wl = synth.WORKLOADS[args.workload]
    st = oracle_setup(wl, args.seed)
    g, q = st["g"], st["q"]
    rhs = lambda x: osw.rhs_real(g, x.reshape(q.shape)).reshape(-1)                       # noqa: E731
    jvp = lambda x, w: osw.jvp(g, x.reshape(q.shape), w.reshape(q.shape)).reshape(-1)     # noqa: E731
    it = oepi.EPI(rhs, jvp, wl.order, tol=wl.tol)
    y = q.reshape(-1).copy()
    Fn = rhs(y)
    P = oepi.history_length(wl.order)
    it.history = [(y - i * wl.dt * Fn, rhs(y - i * wl.dt * Fn)) for i in range(1, P + 1)]
    t0 = time.perf_counter()
    y = it.step(y, wl.dt)
    sec = time.perf_counter() - t0
    k = it.stats[-1]
    print(json.dumps({"oracle_full_step": {
        "workload": wl.name, "order": wl.order, "seconds": sec, "steps_per_s": 1.0 / sec, "cores": 1,
        "krylov_iters": k["krylov_iters"], "attempts": k["substeps"] + k["rejects"], "substeps": k["substeps"],
        "rejects": k["rejects"], "finite": bool(np.all(np.isfinite(y)))}}), flush=True)


def main():
    args = parse()
    if args.oracle_full_step:
        run_oracle_full_step(args)
        return
    if args.kiops_call:
        run_kiops_call(args)
        return
    world, rank, local, pg = dist_setup(args)
    if args.impl == "reference":
        run_reference(args, world, rank)
        if pg is not None:
            pg.barrier()
            pg.destroy_process_group()
        return
    import numpy as np
    import torch

    from paper_2101_05617_gb300 import swepi, synth
    if args.warmup < 3:
        raise SystemExit("--warmup must be >= 3")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    wl = synth.WORKLOADS[args.workload]
    P = {2: 0, 3: 1, 4: 2, 5: 3, 6: 4}[wl.order]
    f = synth.make_fields(wl, args.seed + rank)
    ctx = swepi.SWContext(wl.ne, wl.p, f.rotation)
    h, hB, V = f.evaluate(ctx.node_xyz())
    q_host = ctx.state_from_fields(h, hB, V)
    q = torch.tensor(q_host, device=dev)
    if args.jvp_mode == 2:
        raise SystemExit("--jvp-mode 2 applies to --kiops-call; the timed step is the FP64 path")
    ctx.set_jvp_mode(args.jvp_mode)
    opts = dict(tol=wl.tol)
    stream = torch.cuda.current_stream()

    for _ in range(args.warmup):
        ctx.epi_step(wl.order, wl.dt, q, **opts)
    torch.cuda.synchronize()
    ctl = None
    if args.control == "learned":
        from paper_2101_05617_gb300 import learned
        ctl = learned.Controller.load()
        swepi.sw_set_controller(ctx.handle, ctl.handle)

    gpu_index = os.environ.get("CUDA_VISIBLE_DEVICES", str(local)).split(",")[local if world > 1 else 0]
    clocks = ClockSampler(gpu_index)
    krylov = 0
    krylov_list = []
    attempts = substeps = 0
    if pg is not None:
        pg.barrier()
    torch.cuda.synchronize()
    clocks.start()
    # the dominant kernel alone is bracketed by events in the timed region, one
    # launch in PROFILE_EVERY (an event pair between kernels keeps the next from
    # overlapping the previous one's tail); the other families are timed in a
    # separate step
    ctx.profile_every(PROFILE_EVERY)
    ctx.profile_kinds("volume_jvp")
    launches0 = ctx.kernel_launches()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record(stream)
    for _ in range(args.steps):
        st = ctx.epi_step(wl.order, wl.dt, q, **opts)
        krylov += st["krylov_iters"]
        krylov_list.append(st["krylov_iters"])
        attempts += st["substeps"] + st["rejects"]
        substeps += st["substeps"]
    e1.record(stream)
    torch.cuda.synchronize()
    if pg is not None:
        pg.barrier()
    elapsed_ms = e0.elapsed_time(e1)
    clock_info = clocks.stop()
    launches = ctx.kernel_launches() - launches0
    prof = ctx.profile_read()
    ctx.profile(False)
    max_ms, total_steps = aggregate(pg, elapsed_ms, args.steps, dev if pg is not None else None)

    swepi.sw_set_controller(ctx.handle, None)
    ctx.close()

    # end to end through the public API with host buffers, on a fresh context that
    # replays the same trajectory (same warm-up, then the timed steps): per step the
    # state is copied in from pinned host memory and the result read back.  The last
    # warm-up step of this replay is the breakdown step: every kernel family bracketed
    # by events (outside both timed regions).
    ctx = swepi.SWContext(wl.ne, wl.p, f.rotation)
    ctx.set_jvp_mode(args.jvp_mode)
    fused_main = bool(ctx.set_orth_fused(1))
    q = torch.tensor(q_host, device=dev)
    for k in range(args.warmup):
        if k == args.warmup - 1:
            torch.cuda.synchronize()
            ctx.profile(True)
            b0 = torch.cuda.Event(enable_timing=True)
            b1 = torch.cuda.Event(enable_timing=True)
            b0.record(stream)
        ctx.epi_step(wl.order, wl.dt, q, **opts)
    b1.record(stream)
    torch.cuda.synchronize()
    breakdown_ms = b0.elapsed_time(b1)
    prof_all = ctx.profile_read()
    ctx.profile(False)
    if ctl is not None:
        swepi.sw_set_controller(ctx.handle, ctl.handle)
    q_pin = torch.from_numpy(q.cpu().numpy()).pin_memory()
    if pg is not None:
        pg.barrier()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    for _ in range(args.steps):
        # the C-ABI call on the host state: copy in, one EPI step, copy back
        ctx.epi_step_host(wl.order, wl.dt, q_pin, **opts)
    e2e_s = time.perf_counter() - t0
    e2e_max, _ = aggregate(pg, e2e_s * 1e3, args.steps, dev if pg is not None else None)

    if rank == 0:
        ne, ns = wl.ne, wl.ns
        fv, ff = flops_per_jvp(ne, ns)
        if args.jvp_mode == 0:   # full evaluation per vector: first-order complex arithmetic counts
            fv, ff = 6 * ne * ne * ns * ns * (108 + 12 * ns), 12 * ne * ne * ns * (30 * ns + 182)
        vj, fj = prof["volume_jvp"], prof_all["face_jvp"]
        t_vol = vj["ms"] / max(1, vj["count"]) * 1e-3
        t_face = fj["ms"] / max(1, fj["count"]) * 1e-3
        dominant = "volume" if prof_all["volume_jvp"]["ms"] >= prof_all["face_jvp"]["ms"] else "face"
        # these kernels do most of their arithmetic in block fixed point on the integer pipe, so the FP64 peak is
        # no roofline of theirs: the bytes they must move are
        rpeak, peak_src = hbm_peak_gbs()
        nodes = 6 * ne * ne * ns * ns
        if args.jvp_mode == 0:
            nb = nodes * full_bytes_per_node(ns, dominant, 2, EPI_PHI[wl.order])
        elif dominant == "volume":
            nb = nodes * volume_bytes_per_node(ns, 1, 2, EPI_PHI[wl.order])
        else:
            nb = nodes * face_bytes_per_node(ns)
        achieved = nb / (t_vol if dominant == "volume" else t_face) / 1e9
        peak_src = f"HBM copy bandwidth ({peak_src}); algorithmic bytes {nb:.4g} a launch"
        roofline = {"bound": "hbm", "achieved": achieved, "peak": rpeak, "unit": "GB/s",
                    "frac": achieved / rpeak,
                    "traffic": TRAFFIC_BYTES.get(wl.name) if dominant == "volume" and args.jvp_mode == 1 else None,
                    "kernel": ((f"volume_tangent_kernel<double,{ns}>" if dominant == "volume"
                                else f"face_tangent_kernel<double,{ns}>")
                               + " (imaginary half of the complex-step JVP, phi-solver epilogue)")
                              if args.jvp_mode == 1 else f"{dominant} kernel<cs,{ns}> (full complex-step JVP)",
                    "peak_source": peak_src,
                    "per_kernel": {"volume": {"flops": fv, "avg_ms": t_vol * 1e3, "launches": vj["count"],
                                              "bracketed_every": PROFILE_EVERY,
                                              "tflops": fv / t_vol / 1e12 if t_vol else None},
                                   "face": {"flops": ff, "avg_ms": t_face * 1e3, "launches": fj["count"],
                                            "tflops": ff / t_face / 1e12 if t_face else None},
                                   "expm": {"avg_ms": prof_all["expm"]["ms"] / max(1, prof_all["expm"]["count"]),
                                            "launches": prof_all["expm"]["count"]},
                                   "orthogonalisation": ortho_roofline(prof_all, wl, fused_main)},
                    "share_of_step": {k: prof_all[k]["ms"] / breakdown_ms
                                      for k in ("volume_jvp", "face_jvp", "orthogonalisation", "expm", "linearize")},
                    "share_note": "the last warm-up EPI step of the end-to-end replay with every kernel family "
                                  "bracketed by events; the timed region brackets only the dominant kernel"}
        t_jvp = t_vol + t_face
        value = total_steps / (max_ms * 1e-3)
        out = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
               "warmup": args.warmup, "ms_per_step": max_ms / args.steps, "higher_is_better": True,
               "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
               "config": {"workload": f"{wl.name}: 6x{ne}x{ne} elements, p={wl.p}, EPI{wl.order}, "
                                      f"dt={wl.dt:g} s, KIOPS tol {wl.tol:g}, complex-step eps {wl.eps:g}",
                          "n_unknowns": wl.n_unknowns, "parallelism": "replicas" if world > 1 else "single",
                          "control": args.control,
                          "l2": "inputs larger than L2 (Krylov basis ~2.4 GB per KIOPS call)"},
               "jvp_dof_per_s": wl.n_unknowns / t_jvp,
               "jvp_dof_per_s_total": world * wl.n_unknowns / t_jvp,
               "jvp_nodes_per_s": wl.n_unknowns / 3 / t_jvp,   # the paper's DOF count: one per solution point
               "krylov_iters_per_step": krylov / args.steps,
               "krylov_iters_each_step": krylov_list,
               "substep_attempts_per_step": attempts / args.steps,
               "substeps_per_step": substeps / args.steps,
               "clocks": clock_info,
               "e2e": {"value": total_steps / (e2e_max * 1e-3), "unit": UNIT,
                       "h2d_bytes_per_step": 8 * wl.n_unknowns, "d2h_bytes_per_step": 8 * wl.n_unknowns},
               "gpu_launches": launches,
               "roofline": roofline,
               "forms": {"timed": ("learned control + FP64 split complex-step JVP" if ctl is not None
                                   else "plain control + FP64 split complex-step JVP")}}
        if not args.no_forms and world == 1:   # replicas (N > 1) time the step only
            from paper_2101_05617_gb300 import learned

            only = {x.strip() for x in args.only_forms.split(",") if x.strip()}
            short = {"learned_vs_plain_same_start": "learned", "complex64_bulk_ne30_p5": "ne30",
                     "complex64_bulk_ne60_p5": "ne60", "ensemble_96": "ensemble", "large_ne90_p6": "large"}

            def form(name, fn):
                if only and short[name] not in only:
                    return
                # a form that fails is reported, not allowed to lose the benchmark line
                try:
                    out["forms"][name] = fn()
                except Exception as e:
                    out["forms"][name] = {"error": f"{type(e).__name__}: {e}"[:300]}
                torch.cuda.synchronize()

            lc = ctl if ctl is not None else learned.Controller.load()
            form("learned_vs_plain_same_start",
                 lambda: learned.evaluate(lc, args.workload, args.steps, seed=args.seed + 1))
            # the complex64-bulk form with its orthogonalisation window of three (reading 17) on configuration 2
            form("complex64_bulk_ne30_p5", lambda: fp32_form_comparison(
                args, dev, "ne30_p5", (("fp64", 1, 2), ("complex64_bulk_window3", 2, 3))))
            if args.workload == "ne60_p5":
                # on this grid the form needs the orthogonalisation window of three
                # the configured 48 EPI5 steps of this grid (4 untimed, 44 timed) from the same start
                form("complex64_bulk_ne60_p5", lambda: fp32_form_comparison(
                    args, dev, "ne60_p5", (("fp64", 1, 2), ("fp64_window3", 1, 3), ("complex64_bulk_window3", 2, 3),
                                           ("complex64_bulk_window3_learned", 2, 3, "learned"),
                                           ("fp64_device_controller", 1, 2, "device"),
                                           ("complex64_bulk_window3_device_controller", 2, 3, "device")),
                    per_kernel=True, total_steps=48))
            if world == 1 and not args.no_ensemble:
                form("ensemble_96", lambda: ensemble_form(args, dev))
            if world == 1 and not args.no_large:
                # the large single instance: 6 x 90 x 90 elements, p = 6, bottom topography, EPI6 over its
                # configured 36 steps at dt = 600 s: at the configured 1200 s (and at 900 s) the FP64 method
                # itself goes unstable within the 36 steps (the order-6 vorticity growth), at 600 s both
                # forms stay finite
                form("large_ne90_p6", lambda: fp32_form_comparison(
                    args, dev, "ne90_p6", (("fp64", 1, 2), ("complex64_bulk_window3", 2, 3)), per_kernel=True,
                    total_steps=36, dt=LARGE_STABLE_DT))
        if world == 1 and not args.no_cpu_baseline:
            counts = (krylov / args.steps, attempts / args.steps, substeps / args.steps)
            out["cpu_baseline"] = oracle_sample(wl, args.seed, counts, P)
            out["cpu_baseline_all_cores"] = oracle_sample_all_cores(wl, args.seed, krylov / args.steps, P,
                                                                    out["cpu_baseline"])
        out["headline"] = headline(out)
        print(json.dumps(out), flush=True)
    swepi.sw_set_controller(ctx.handle, None)
    ctx.close()
    if pg is not None:
        pg.barrier()
        pg.destroy_process_group()


if __name__ == "__main__":
    main()
