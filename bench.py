"""Benchmark: solution-point RK-stage updates/s of the FR residual + RK44 stage update.

Workload: Taylor-Green vortex (Ma 0.1, Re 1600) on a periodic 64^3 hexahedral mesh at p = 4
(125 Gauss-Legendre points per element, 32.8 M solution points, 164 M unknowns), compressible
Navier-Stokes with Rusanov + BR2 fluxes and the DG-equivalent correction.  The headline value is
the double-float path (FR_PREC_MIXED); the same path with its viscous branch in FP32
(FR_PREC_MIXED_VF32) and the FP64 path are reported beside it.
One step = one RK44 time step = 4 RK stages (each: residual + stage update); the metric counts
solution points x stages per second.  Inputs are synthetic and seeded; the device working set
(~18 GB) is far larger than L2, so no flush is needed between iterations.

Prints one JSON line of at most 1500 characters with the headline, the end-to-end rate and the p = 3..7 rates
(`headline`); --detail FILE writes everything that was measured.

Usage: python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference] [--detail FILE]
Under torchrun (N > 1) every rank runs an independent replica on its own GPU (weak scaling by
replicas; the domain-decomposed stage with halo exchange, fr_part_phase, is not timed across GPUs
here), timing is max over ranks.
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

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

METRIC = "solution-pt RK-stage updates/s at p=3..7, mixed-prec vs FP64, at stated error"
UNIT = "updates/s"
N_EDGE, ORDER, CFL = 64, 4, 0.3


def config(precision="fp64"):
    n_pts = N_EDGE ** 3 * (ORDER + 1) ** 3
    return {"workload": f"tgv_{N_EDGE}cube_p{ORDER}_{precision}", "mesh": f"{N_EDGE}^3 periodic hex [0,2pi]^3", "p": ORDER,
            "n_points": n_pts, "unknowns": 5 * n_pts, "case": "TGV Ma=0.1 Re=1600 gamma=1.4 Pr=0.71",
            "flux": "Rusanov + BR2, VCJH c=0 (DG)", "integrator": "RK44, CFL 0.3", "precision": precision,
            "l2": "no flush: working set ~18 GB >> 129 MB L2"}


def _env_rank():
    return int(os.environ.get("RANK", "0")), int(os.environ.get("WORLD_SIZE", "1")), int(os.environ.get("LOCAL_RANK", "0"))


def _dist_barrier(world):
    """Barrier over the replicas (no-op for one process)."""
    if world > 1:
        import torch.distributed as dist
        dist.barrier()


def _dist_max(v, world, device):
    """Max of a timing scalar over the replicas (all-reduce of one number; no data-path exchange)."""
    if world > 1:
        import torch
        import torch.distributed as dist
        tt = torch.tensor([v], device=device, dtype=torch.float64)
        dist.all_reduce(tt, op=dist.ReduceOp.MAX)
        v = float(tt.item())
    return v


# ------------------------------------------------------------------------------ clocks sampling
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_id: str):
        self.gpu_id = gpu_id
        self.proc = None
        self.path = None

    def start(self):
        try:
            fd, self.path = tempfile.mkstemp(suffix=".csv")
            os.close(fd)
            self.proc = subprocess.Popen(["nvidia-smi", "-i", self.gpu_id, f"--query-gpu={self.FIELDS}",
                                          "--format=csv,noheader,nounits", "-lms", "200", "-f", self.path],
                                         stdout=subprocess.DEVNULL, stderr=subprocess.DEVNULL)
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
        rows = []
        try:
            with open(self.path) as fh:
                for line in fh:
                    parts = [s.strip() for s in line.split(",")]
                    if len(parts) >= 9:
                        rows.append(parts)
            os.unlink(self.path)
        except Exception:
            pass
        if not rows:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["no samples"]}
        sm = [float(r[1]) for r in rows if r[1].replace(".", "").isdigit()]
        mx = [float(r[2]) for r in rows if r[2].replace(".", "").isdigit()]
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = sorted({names[k] for r in rows for k in range(4) if r[5 + k].lower().startswith("active")})
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": reasons, "samples": len(rows)}


# ------------------------------------------------------------------------------ CPU oracle timing
def oracle_rate(budget_s=12.0, max_steps=None, n=8, p=ORDER):
    """Time the oracle (as it stands) on an n^3, order-p periodic TGV: RK44 steps until the
    budget is used.  Returns (updates/s, sample description, threads used)."""
    from oracle.hexfr import HexFR
    from paper_2308_06605_gb300 import inputs as I
    m = HexFR(I.hex_box_mesh((n, n, n)), I.tgv_physics(), p)
    Q = I.tgv_state(m.x)
    dt = m.max_dt(Q, CFL)
    steps, t0 = 0, time.perf_counter()
    while True:
        Q = m.rk44_step(Q, 0.0, dt)
        steps += 1
        el = time.perf_counter() - t0
        if (max_steps and steps >= max_steps) or (not max_steps and el >= budget_s):
            break
    rate = m.E * m.Np * 4 * steps / el
    return rate, f"oracle RK44 on {n}^3 hex p={p} TGV ({m.E * m.Np} points), {steps} steps in {el:.1f} s", 1


def _oracle_worker(budget_s):
    return oracle_rate(budget_s=budget_s)[:2]


def oracle_rate_procs(budget_s=12.0, procs=1):
    """The oracle as it stands in `procs` spawned processes at once, one independent replica of
    the same workload each, BLAS and OpenMP threads pinned to 1 so a replica uses one core.
    Returns (aggregate updates/s, sample of one replica, processes)."""
    import multiprocessing as mp
    keys = ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS")
    saved = {k: os.environ.get(k) for k in keys}
    for k in keys:
        os.environ[k] = "1"
    try:
        with mp.get_context("spawn").Pool(procs) as pool:
            res = pool.map(_oracle_worker, [budget_s] * procs)
    finally:
        for k, v in saved.items():
            if v is None:
                os.environ.pop(k, None)
            else:
                os.environ[k] = v
    return sum(r for r, _ in res), res[0][1], procs


def run_reference(args):
    rank, world, _ = _env_rank()
    if rank != 0:
        return 0
    # One core, as reported: BLAS / OpenMP threads pinned before NumPy is first imported.
    for k in ("OMP_NUM_THREADS", "OPENBLAS_NUM_THREADS", "MKL_NUM_THREADS"):
        os.environ.setdefault(k, "1")
    for _ in range(args.warmup):
        oracle_rate(max_steps=1)
    t0 = time.perf_counter()
    rate, sample, cores = oracle_rate(max_steps=args.steps)
    el = time.perf_counter() - t0
    cfg = dict(config("mixed"))
    cfg["reference_sample"] = ("each step: one oracle RK44 step on the 8^3 periodic hex TGV at p=4 (64 000 points; "
                               "same case, order and per-point work as the 64^3 workload, 1/512 of its points)")
    line = {"impl": "reference", "metric": METRIC, "value": rate, "unit": UNIT, "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * el / max(1, args.steps),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64",
            "data": "synthetic", "config": cfg,
            "cpu_baseline": {"value": rate, "unit": UNIT, "cores": cores, "kind": "oracle", "sample": sample},
            "e2e": {"value": rate, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)
    return 0


# ------------------------------------------------------------------------------ GPU path
SWEEP = [(64, 3), (64, 4), (48, 5), (40, 6), (32, 7)]   # (elements per edge, p): 17-33 M points
# A term of a compensated double-float sum (2 algorithmic flops) is 12 FP32 instructions (4 for the
# product with its error and cross terms, 6 for the sum with its error, 2 to collect the errors); the FP32 peak in
# FLOP/s counts an FFMA instruction as 2 flops, so the double-float peak in algorithmic FLOP/s is
# fp32_peak / 2 instructions/s * 2 / 12 = fp32_peak / 12.
DF_FP32_FLOPS_PER_FLOP = 12.0


class Case:
    """One mesh + state on the device, stepping with RK44 on the torch current stream."""

    def __init__(self, n_edge, p, precision, dt=None, prisms=None, vcjh_c=0.0):
        import numpy as np
        import torch
        from paper_2308_06605_gb300 import fr, inputs as I
        self.torch = torch
        self.stream = torch.cuda.current_stream()
        phys = I.tgv_physics()
        phys.precision = {"fp64": 0, "mixed": 1, "mixed_tc": 2, "mixed_vf32": 3}[precision]
        phys.vcjh_c = vcjh_c
        self.mesh = fr.Mesh(I.hex_box_mesh((n_edge, n_edge, n_edge), prisms=prisms), phys, p,
                            stream=self.stream.cuda_stream)
        x = self.mesh.solution_points()
        self.Q0 = np.ascontiguousarray(I.tgv_state(x, Ma=0.1))
        del x
        self.Qd = torch.from_numpy(self.Q0).to("cuda")
        self.mesh.set_state(self.Qd)
        self.dt = dt if dt is not None else self.mesh.max_dt(CFL)
        self.n_pts = self.mesh.n_points
        self.t = 0.0

    def step(self):
        for s in range(4):
            self.mesh.rk_stage(s, self.t, self.dt)
        self.t += self.dt

    def timed(self, steps):
        torch = self.torch
        torch.cuda.synchronize()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record(self.stream)
        for _ in range(steps):
            self.step()
        e1.record(self.stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1)

    def kernels(self, steps, p, prism_model=False):
        from paper_2308_06605_gb300 import perfmodel
        self.mesh.profile(True)
        for _ in range(steps):
            self.step()
        kms, kcnt = self.mesh.profile_read(4)
        self.mesh.profile(False)
        if prism_model:
            fl, by = perfmodel.prism_flops_per_point(p), perfmodel.prism_bytes_per_point(p)
        else:
            fl, by = perfmodel.flops_per_point(p), perfmodel.bytes_per_point(p)
        out = {}
        for k, name in enumerate(perfmodel.KERNELS):
            avg = kms[k] / max(1, kcnt[k])
            out[name] = {"launches": kcnt[k], "avg_ms": avg, "share": kms[k] / max(1e-30, sum(kms)),
                         "gflops": fl[name] * self.n_pts / (avg * 1e-3) / 1e9 if avg > 0 else None,
                         "gbs": by[name] * self.n_pts / (avg * 1e-3) / 1e9 if avg > 0 else None}
        return out

    def close(self):
        self.mesh.close()
        del self.Qd


def run_ensemble(precision, steps, stream):
    """The 64-case isentropic-vortex ensemble (n^3 periodic hexes, n ~ U{8..24}, p ~ U{2..5},
    Ma 0.5, beta 5, centres from splitmix64; Euler) advanced by one persistent launch per RK
    stage (fr_batch), after autotuning; compared with launching every case's kernels per stage."""
    import numpy as np
    import torch
    from paper_2308_06605_gb300 import fr, inputs as I
    cases = I.vortex_ensemble(64)
    meshes, dts = [], []
    for c in cases:
        L = c["L"]
        d = I.hex_box_mesh((c["n"],) * 3, lo=(-L / 2,) * 3, hi=(L / 2,) * 3)
        ph = I.Physics(gamma=1.4, R=1.0, mu=0.0, viscous=0, precision=1 if precision == "mixed" else 0)
        m = fr.Mesh(d, ph, c["p"], stream=stream.cuda_stream)
        x = m.solution_points()
        m.set_state(np.ascontiguousarray(I.isentropic_vortex_state(x, centre=c["centre"], period=(L, L))))
        dts.append(m.max_dt(CFL))
        meshes.append(m)
    n_pts = sum(m.n_elem * m.n_pts for m in meshes)
    out = {"cases": len(meshes), "n_points": n_pts, "orders": sorted({c["p"] for c in cases})}

    def timed(fn, k):
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record(stream)
        for _ in range(k):
            fn()
        e1.record(stream)
        torch.cuda.synchronize()
        return e0.elapsed_time(e1) / k

    def per_mesh_step():
        for s_ in range(4):
            for m, dt in zip(meshes, dts):
                m.rk_stage(s_, 0.0, dt)
    per_mesh_step()
    out["per_mesh_launches_updates_per_s"] = n_pts * 4 / (timed(per_mesh_step, steps) * 1e-3)
    with fr.Batch(meshes) as b:
        b.tune()
        b.set_dt(dts)
        b.rk_step()
        ms = timed(b.rk_step, steps)
        out["updates_per_s"] = n_pts * 4 / (ms * 1e-3)
        out["ms_per_step"] = ms
        out["tuned"] = b.info()
        chosen = out["tuned"]["mode"]
        for mode, key in ((0, "persistent_updates_per_s"), (1, "per_case_graph_updates_per_s")):
            b.select(mode)
            b.rk_step()
            out[key] = n_pts * 4 / (timed(b.rk_step, steps) * 1e-3)
        b.select(chosen)
    for m in meshes:
        m.close()
    return out


PRISM_CASES = [(48, 4, "all"), (48, 4, "checker"), (24, 7, "all")]   # (edge, p, split): 11-22 M points


def run_prisms(steps, fp64_peak, df_peak, cases=None):
    """Prismatic and mixed hexahedral/prismatic periodic TGV meshes, both precisions: updates/s,
    and on the all-prism meshes the phase times with the prism cost model and the volume kernel's
    fraction of the arithmetic peak."""
    out = {}
    for (n, p, split) in (cases or PRISM_CASES):
        row = {"n_edge": n, "p": p, "split": split}
        dt = None
        for prec in ("fp64", "mixed"):
            c = Case(n, p, prec, dt=dt, prisms=split)
            dt = c.dt
            row["n_points"] = c.n_pts
            row["n_prism"], row["n_hex"] = c.mesh.n_prism, c.mesh.n_elem
            c.step()
            ms = c.timed(max(2, steps))
            row[prec] = c.n_pts * 4 * max(2, steps) / (ms * 1e-3)
            if split == "all":
                k = c.kernels(2, p, prism_model=True)
                peak = fp64_peak if prec == "fp64" else df_peak
                row[prec + "_kernels"] = k
                row[prec + "_volume_frac_of_peak"] = k["volume"]["gflops"] * 1e9 / peak
            c.close()
        out[f"{split}_{n}cube_p{p}"] = row
    return out


def run_tc(steps, n=N_EDGE, p=ORDER):
    """The double-float path with the face interpolation on the tensor cores (FR_PREC_MIXED_TC)
    against the plain double-float path on the benchmark mesh: RK44 updates/s, the face
    interpolation's time per stage, and each residual's error against the FP64 path."""
    row = {"n_edge": n, "p": p, "n_points": n ** 3 * (p + 1) ** 3}
    c64 = Case(n, p, "fp64")
    dt = c64.dt
    for tag, prec in (("mixed", "mixed"), ("mixed_tc", "mixed_tc")):
        c = Case(n, p, prec, dt=dt)
        row[tag + "_error_vs_fp64"] = residual_error(c, c64)
        c.step()
        ms = c.timed(max(2, steps))
        row[tag] = c.n_pts * 4 * max(2, steps) / (ms * 1e-3)
        k = c.kernels(2, p)
        row[tag + "_interp_ms"] = k["interp_faces"]["avg_ms"]
        row[tag + "_interp_gbs"] = k["interp_faces"]["gbs"]
        c.close()
    c64.close()
    return row


def run_vcjh(steps, n=48, p=4):
    """Correction function c_HU (energy-stable family, Huynh's g2) against the DG-equivalent c = 0
    on the TGV box, both precisions: updates/s of RK44 steps."""
    import math
    apf = math.factorial(2 * p) / (2.0 ** p * math.factorial(p))
    c_hu = 2.0 * (p + 1) / ((2 * p + 1) * p * apf ** 2)
    row = {"n_edge": n, "p": p, "c": c_hu, "n_points": n ** 3 * (p + 1) ** 3}
    for prec in ("fp64", "mixed"):
        dt = None
        for tag, c in (("c0", 0.0), ("c_hu", c_hu)):
            cs = Case(n, p, prec, dt=dt, vcjh_c=c)
            dt = cs.dt
            cs.step()
            ms = cs.timed(max(2, steps))
            row[f"{prec}_{tag}"] = cs.n_pts * 4 * max(2, steps) / (ms * 1e-3)
            cs.close()
    return row


def run_cascade(steps, fp64_peak, df_peak, nz=40, p=7):
    """The synthetic cascade passage (398 000 quadratic elements at nz = 40, 24 % prisms, p = 7,
    182 M points): walls, characteristic inflow/outflow, periodic pitch and span; both precisions,
    RK44 steps at the stable step from the seeded inflow state; updates/s and the phase times."""
    import numpy as np
    import torch
    from paper_2308_06605_gb300 import fr, inputs as I
    out = {}
    stream = torch.cuda.current_stream()
    dt = None
    for prec in ("fp64", "mixed"):
        phys, bcs, state_fn = I.cascade_conditions()
        phys.precision = 1 if prec == "mixed" else 0
        d = I.blade_passage_mesh(nz=nz, bcs=bcs)
        t0 = time.perf_counter()
        m = fr.Mesh(d, phys, p, stream=stream.cuda_stream)
        t_create = time.perf_counter() - t0
        x = m.solution_points()
        Qd = torch.from_numpy(np.ascontiguousarray(state_fn(x, perturb=1e-3))).to("cuda")
        del x
        m.set_state(Qd)
        if dt is None:
            # RK44 with dt = CFL h / ((2p+1) lambda) is unstable for p >= 5; the stable step scales
            # like h / ((p+1)^2 lambda), so the CFL number is rescaled by (2p+1)/(p+1)^2.
            dt = m.max_dt(0.3 * (2 * p + 1) / (p + 1) ** 2)
        for _ in range(2):
            m.rk_step(0.0, dt)
        torch.cuda.synchronize()
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        k = max(2, steps)
        e0.record(stream)
        for _ in range(k):
            m.rk_step(0.0, dt)
        e1.record(stream)
        torch.cuda.synchronize()
        ms = e0.elapsed_time(e1) / k
        m.profile(True)
        m.rk_step(0.0, dt)
        kms, kcnt = m.profile_read(4)
        m.profile(False)
        out[prec] = {"updates_per_s": m.n_points * 4 / (ms * 1e-3), "ms_per_step": ms, "mesh_create_s": t_create,
                     "phase_ms_per_stage": dict(zip(("interp_faces", "volume", "iface_flux", "correct"),
                                                    [a / max(1, c) for a, c in zip(kms, kcnt)]))}
        out["n_points"], out["n_hex"], out["n_prism"], out["p"] = m.n_points, m.n_elem, m.n_prism, p
        out["device_bytes_" + prec] = m.device_bytes
        m.close()
        del Qd
        torch.cuda.empty_cache()
    out["dt"] = dt
    return out


def residual_error(a, b):
    """Per-variable max-norm and L2 relative difference of two device residuals (b = reference)."""
    torch = a.torch
    Ra = torch.empty_like(a.Qd)
    Rb = torch.empty_like(b.Qd)
    a.mesh.set_state(a.Qd)
    b.mesh.set_state(b.Qd)
    a.mesh.residual(out=Ra)
    b.mesh.residual(out=Rb)
    torch.cuda.synchronize()
    d = (Ra - Rb).reshape(-1, 5)
    r = Rb.reshape(-1, 5)
    linf = (d.abs().amax(0) / r.abs().amax(0)).tolist()
    l2 = (d.norm(dim=0) / r.norm(dim=0)).tolist()
    names = ["rho", "rho_u", "rho_v", "rho_w", "E"]
    return {"max_rel": dict(zip(names, linf)), "l2_rel": dict(zip(names, l2))}


def run_ours(args):
    import torch
    rank, world, local = _env_rank()
    if world > 1:
        import torch.distributed as dist
        torch.cuda.set_device(local)
        dist.init_process_group("nccl")
    dev = torch.cuda.current_device()
    from paper_2308_06605_gb300 import fr, perfmodel
    if not os.path.exists(fr.LIB_PATH):
        from paper_2308_06605_gb300 import build as B
        B.build()
    fr.load()
    if args.cascade_only:
        print(json.dumps({"cascade_p7": run_cascade(args.steps, None, None)}), flush=True)
        return 0
    if args.tc_only:
        print(json.dumps({"tensor_core_interp": run_tc(args.steps, N_EDGE, ORDER)}), flush=True)
        return 0

    def barrier():
        _dist_barrier(world)

    def max_over_ranks(v):
        return _dist_max(v, world, f"cuda:{dev}")

    # Headline workload: every precision on the same initial state and the same dt.  The headline
    # value is the double-float path (FR_PREC_MIXED, within the error target); the same path with
    # its viscous branch in FP32 (FR_PREC_MIXED_VF32, faster, with a larger error at this viscous-
    # dominated initial state) and the FP64 path are reported beside it.
    c64 = Case(N_EDGE, ORDER, "fp64")
    cmx = Case(N_EDGE, ORDER, "mixed", dt=c64.dt)
    cvf = Case(N_EDGE, ORDER, "mixed_vf32", dt=c64.dt)
    err = residual_error(cmx, c64)
    err_vf = residual_error(cvf, c64)
    n_pts = c64.n_pts
    for c in (c64, cmx, cvf):
        for _ in range(args.warmup):
            c.step()
    props = torch.cuda.get_device_properties(dev)
    uuid = getattr(props, "uuid", None)
    gid = f"GPU-{uuid}" if uuid is not None and not str(uuid).startswith("GPU-") else (str(uuid) if uuid else str(dev))
    sampler = ClockSampler(gid)
    barrier()
    torch.cuda.synchronize()
    sampler.start()
    time.sleep(0.3)
    ms_vf = max_over_ranks(cvf.timed(args.steps))
    ms_mx = max_over_ranks(cmx.timed(args.steps))
    ms_64 = max_over_ranks(c64.timed(args.steps))
    barrier()
    clocks = sampler.stop()
    value = world * n_pts * 4 * args.steps / (ms_mx * 1e-3)
    value_vf = world * n_pts * 4 * args.steps / (ms_vf * 1e-3)
    value64 = world * n_pts * 4 * args.steps / (ms_64 * 1e-3)
    k_vf = cvf.kernels(args.steps, ORDER)
    k_mx = cmx.kernels(args.steps, ORDER)
    k_64 = c64.kernels(args.steps, ORDER)
    fp64_peak = fr.probe_fma(0, 4000)
    fp32_peak = fr.probe_fma(1, 200000)
    df_peak = fp32_peak / DF_FP32_FLOPS_PER_FLOP
    fl = perfmodel.flops_per_point(ORDER)
    by = perfmodel.bytes_per_point(ORDER)

    def mixed_roofline(k, fp32_viscous, tag):
        dom = max(k, key=lambda n_: k[n_]["share"])
        peak = perfmodel.mixed_alu_peak(ORDER, df_peak, fp32_peak, fp32_viscous) if dom == "volume" else df_peak
        ach = k[dom]["gflops"] * 1e9
        src = ("measured FP32 FMA rate (fr_probe_fma) / 12 (a term of a compensated double-float sum is 12 FP32 "
               "instructions for 2 algorithmic flops)")
        if fp32_viscous and dom == "volume":
            src = ("the kernel's arithmetic mix at measured rates: the viscous branch's flops at the FP32 FMA rate, "
                   "the rest at that rate / 12 (times added)")
        return {"bound": "alu", "kernel": dom, "precision": tag, "achieved": ach / 1e12, "peak": peak / 1e12,
                "unit": "TFLOP/s", "frac": ach / peak, "traffic": None,
                "peak_source": src, "algorithmic_flops_per_point": fl[dom], "algorithmic_bytes_per_point": by[dom]}

    roofline = mixed_roofline(k_mx, False, "mixed")
    fp32_viscous = {"value": value_vf, "ms_per_step": ms_vf / args.steps, "kernels": k_vf,
                    "roofline": mixed_roofline(k_vf, True, "mixed_vf32"), "error_vs_fp64": err_vf}
    dom64 = max(k_64, key=lambda n_: k_64[n_]["share"])
    fp64 = {"value": value64, "ms_per_step": ms_64 / args.steps, "kernels": k_64,
            "roofline": {"bound": "alu", "kernel": dom64, "achieved": k_64[dom64]["gflops"] / 1e3,
                         "peak": fp64_peak / 1e12, "unit": "TFLOP/s", "frac": k_64[dom64]["gflops"] * 1e9 / fp64_peak,
                         "traffic": None,
                         "peak_source": "measured FP64 DFMA rate (fr_probe_fma)"}}
    c64.close()

    # End to end through the public API with host buffers (headline path): set_state from pinned
    # host memory, four stages, get_state back to pinned host memory, every step.
    cvf.close()
    Qh = torch.from_numpy(cmx.Q0).pin_memory()
    Out = torch.empty_like(Qh).pin_memory()
    k_e2e = max(1, args.steps)
    # W untimed passes first: the first transfers from freshly pinned buffers pay one-time costs.
    for _ in range(max(1, args.warmup)):
        cmx.mesh.set_state(Qh)
        cmx.step()
        cmx.mesh.get_state(out=Out)
    torch.cuda.synchronize()
    # Three timed runs of K steps; the median run is reported (the host<->device copies share the
    # host's memory system with other work, so single runs vary), every run's rate is listed.
    runs = []
    for _rep in range(3):
        barrier()
        phase = [0.0, 0.0, 0.0]          # host wall time of set_state, the four stages, get_state
        phase_min = [1e30, 1e30, 1e30]
        te0 = time.perf_counter()
        for _ in range(k_e2e):
            t0 = time.perf_counter()
            cmx.mesh.set_state(Qh)        # returns after the host buffer has been read
            t1 = time.perf_counter()
            cmx.step()                    # the last stage reads the non-finite flag back (synchronises)
            t2 = time.perf_counter()
            cmx.mesh.get_state(out=Out)   # returns after the result is in host memory
            t3 = time.perf_counter()
            for k_, dtk in enumerate((t1 - t0, t2 - t1, t3 - t2)):
                phase[k_] += dtk
                phase_min[k_] = min(phase_min[k_], dtk)
        torch.cuda.synchronize()
        te = max_over_ranks(time.perf_counter() - te0)
        runs.append((world * n_pts * 4 * k_e2e / te, phase, phase_min))
    runs.sort(key=lambda r: r[0])
    e2e_value, phase, phase_min = runs[len(runs) // 2]
    # Plain copy rates of the same pinned buffers (context for the end-to-end number).
    Qd = torch.empty(Qh.shape, dtype=Qh.dtype, device="cuda")
    rates = {}
    for name, dst, src in (("h2d_gbs", Qd, Qh), ("d2h_gbs", Out, Qd)):
        best = 0.0
        for _ in range(3):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            dst.copy_(src, non_blocking=True)
            torch.cuda.synchronize()
            best = max(best, Qh.numel() * 8 / (time.perf_counter() - t0) / 1e9)
        rates[name] = best
    del Qd
    e2e = {"value": e2e_value, "unit": UNIT, "runs": [r[0] for r in runs], "steps_per_run": k_e2e,
           "h2d_bytes_per_step": int(Qh.numel() * 8), "d2h_bytes_per_step": int(Out.numel() * 8),
           "copy_rates_gbs": rates,
           "phase_ms_per_step": {"set_state": 1e3 * phase[0] / k_e2e, "stages": 1e3 * phase[1] / k_e2e,
                                 "get_state": 1e3 * phase[2] / k_e2e},
           "phase_ms_min": {"set_state": 1e3 * phase_min[0], "stages": 1e3 * phase_min[1],
                            "get_state": 1e3 * phase_min[2]}}
    cmx.close()
    del Qh, Out

    prisms = {}
    if not args.no_prisms:
        cases = [(args.prism_edge, args.prism_order, "all")] if args.prism_edge else None
        prisms = run_prisms(args.steps, fp64_peak, df_peak, cases)

    vcjh = run_vcjh(args.steps) if not args.no_vcjh else {}
    tc_row = run_tc(args.steps) if not args.no_tc else {}

    ensemble = {}
    if not args.no_ensemble:
        es = torch.cuda.Stream()
        with torch.cuda.stream(es):
            for prec in ("fp64", "mixed"):
                ensemble[prec] = run_ensemble(prec, max(2, args.steps), es)

    sweep = {}
    if not args.no_sweep:
        for (n, p) in SWEEP:
            row = {"n_edge": n, "n_points": n ** 3 * (p + 1) ** 3}
            dt = None
            for prec in ("fp64", "mixed", "mixed_vf32"):
                c = Case(n, p, prec, dt=dt)
                dt = c.dt
                c.step()
                ms = c.timed(2)
                row[prec] = n ** 3 * (p + 1) ** 3 * 4 * 2 / (ms * 1e-3)
                # Per-kernel CUDA-event times and each kernel's fraction of the arithmetic peak of
                # its precision (FP64: the DFMA rate; double-float: the FP32 FMA rate / 12; the
                # volume kernel with the viscous branch in FP32: its arithmetic mix at those rates).
                peak = fp64_peak if prec == "fp64" else df_peak
                k = c.kernels(2, p)
                row[prec + "_kernels"] = {name: {"avg_ms": v["avg_ms"], "share": v["share"],
                                                 "frac_of_alu_peak": v["gflops"] * 1e9 / peak if v["gflops"] else None}
                                          for name, v in k.items()}
                vpeak = perfmodel.mixed_alu_peak(p, df_peak, fp32_peak, True) if prec == "mixed_vf32" else peak
                if prec == "mixed_vf32":
                    row[prec + "_kernels"]["volume"]["frac_of_alu_peak"] = k["volume"]["gflops"] * 1e9 / vpeak
                row[prec + "_volume_frac"] = k["volume"]["gflops"] * 1e9 / vpeak
                if prec != "mixed_vf32":
                    row[prec + "_step_frac"] = (sum(perfmodel.flops_per_point(p).values()) * row[prec] / peak)
                c.close()
            sweep[f"p{p}"] = row

    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_mx / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32x2+f64", "data": "synthetic",
            "config": config("mixed"), "clocks": clocks, "e2e": e2e,
            "gpu_launches": 4 * 4 * args.steps, "roofline": roofline, "kernels": k_mx,
            "error_vs_fp64": err, "fp32_viscous_branch": fp32_viscous, "fp64": fp64, "p_sweep_updates_per_s": sweep,
            "ensemble_64_vortex": ensemble, "prisms_tgv": prisms, "vcjh_hu_48cube_p4": vcjh,
            "tensor_core_interp_64cube_p4": tc_row,
            "fp64_fma_peak_tflops": fp64_peak / 1e12, "fp32_fma_peak_tflops": fp32_peak / 1e12}
    if args.cascade:
        line["cascade_p7"] = run_cascade(args.steps, fp64_peak, df_peak)
    if rank == 0 and world == 1 and not args.no_cpu_baseline:
        r1, sample1, _ = oracle_rate_procs(12.0, 1)
        ncpu = os.cpu_count() or 1
        rn, sample, cores = oracle_rate_procs(12.0, ncpu)
        line["cpu_baseline"] = {"value": rn, "unit": UNIT, "cores": cores, "kind": "oracle",
                                "sample": f"{cores} replicas at once, one per host core, each: {sample}",
                                "single_thread": {"value": r1, "unit": UNIT, "cores": 1, "sample": sample1}}
        # The small benchmark case in full (8^3 hexahedra, p = 3, 10 RK44 steps) and one RK44 step
        # per order on 4^3 meshes (the oracle's dense operators make larger sweeps take minutes).
        r_c1, s_c1, _ = oracle_rate(max_steps=10, n=8, p=3)
        line["cpu_baseline"]["tgv_8cube_p3_10_steps"] = {"value": r_c1, "unit": UNIT, "cores": 1, "sample": s_c1}
        line["cpu_baseline"]["p_sweep_4cube"] = {}
        for (_, pp) in SWEEP:
            r_p, s_p, _ = oracle_rate(max_steps=1, n=4, p=pp)
            line["cpu_baseline"]["p_sweep_4cube"][f"p{pp}"] = {"value": r_p, "unit": UNIT, "cores": 1, "sample": s_p}
    if world > 1:
        torch.distributed.destroy_process_group()
    if rank == 0:
        if args.detail:
            with open(args.detail, "w") as fh:
                json.dump(line, fh)
        print(json.dumps(headline(line)), flush=True)
    return 0


def headline(full):
    """The printed line: the contract's keys and the rates of every order and precision, in at most 1500
    characters (records of a run keep the end of its output; a longer line was cut and lost)."""
    def digits(x, n):
        return float(f"{x:.{n}g}") if isinstance(x, float) else x

    keys = ("metric", "value", "unit", "n_gpus", "steps", "warmup", "ms_per_step", "higher_is_better", "scaling",
            "vs_baseline", "dtype", "data", "config", "clocks")
    out = {k: digits(full[k], 7) for k in keys}
    out["e2e"] = {k: digits(full["e2e"][k], 7) for k in ("value", "unit", "h2d_bytes_per_step", "d2h_bytes_per_step")}
    out["gpu_launches"] = full["gpu_launches"]
    out["roofline"] = {k: digits(full["roofline"][k], 4) for k in ("bound", "kernel", "achieved", "peak", "unit", "frac")}
    out["l2_error_vs_fp64"] = digits(max(full["error_vs_fp64"]["l2_rel"].values()), 3)
    # [FP64, double-float, FP32 viscous branch]
    out["updates_per_s"] = {f"p{ORDER}": [digits(v, 4) for v in (full["fp64"]["value"], full["value"],
                                                               full["fp32_viscous_branch"]["value"])]}
    for p, row in full["p_sweep_updates_per_s"].items():
        out["updates_per_s"].setdefault(p, [digits(row[k], 4) for k in ("fp64", "mixed", "mixed_vf32")])
    if "cpu_baseline" in full:
        out["cpu_baseline"] = {k: digits(full["cpu_baseline"][k], 5) for k in ("value", "unit", "cores", "kind")}
        out["cpu_baseline"]["sample"] = "oracle RK44, 8^3 hex p=4 TGV, one replica per core"
    return out


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=5)
    ap.add_argument("--warmup", type=int, default=3)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--detail", default="", help="write everything that was measured to this file (JSON)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-sweep", action="store_true", help="skip the p = 3..7 sweep")
    ap.add_argument("--no-ensemble", action="store_true", help="skip the 64-case batched vortex ensemble")
    ap.add_argument("--no-prisms", action="store_true", help="skip the prismatic / mixed-mesh measurements")
    ap.add_argument("--no-vcjh", action="store_true", help="skip the c != 0 correction-function measurement")
    ap.add_argument("--prism-edge", type=int, default=0, help="only an all-prism box of this edge (profiling)")
    ap.add_argument("--prism-order", type=int, default=4)
    ap.add_argument("--cascade", action="store_true",
                    help="also run the synthetic cascade passage (398 000 quadratic elements, p = 7, 182 M points)")
    ap.add_argument("--cascade-only", action="store_true", help="print only the cascade measurement")
    ap.add_argument("--no-tc", action="store_true", help="skip the tensor-core face-interpolation measurement")
    ap.add_argument("--tc-only", action="store_true",
                    help="print only the tensor-core face-interpolation measurement (with --n-edge / --order)")
    ap.add_argument("--n-edge", type=int, default=N_EDGE, help="elements per edge (profiling of smaller cases)")
    ap.add_argument("--order", type=int, default=ORDER)
    args = ap.parse_args()
    globals()["N_EDGE"], globals()["ORDER"] = args.n_edge, args.order
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
