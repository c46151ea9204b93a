#!/usr/bin/env python3
"""Benchmark of the FSLBM time step (stream-collide, free boundary, mass
exchange, conversion, LSQR curvature) on the 256^3 oscillating droplet.

Prints one JSON line (rank 0).  `value` is whole-job fluid-cell updates per
second (MLUPS over liquid + interface cells) with the state resident in HBM;
each timed step is bracketed by CUDA events on the launching stream and L2 is
flushed (256 MiB write) before every step, outside the timed interval.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl fsl|reference]

Multi-GPU: one process per GPU (torchrun); every rank advances an independent
replica (its own seeded droplet), so the work per GPU is fixed (weak scaling)
and there is no data-path collective; only the timing is reduced (max).
`--impl reference` times the FP64 CPU oracle on a bounded sample of the same
workload (the droplet cropped to its bounding box) on the host cores.
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "FSLBM MLUPS & curvature evals/s at 256^3 at stated κ error vs FP64 oracle"
L2_FLUSH_BYTES = 256 << 20


def parse():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=1000)
    ap.add_argument("--warmup", type=int, default=20)
    ap.add_argument("--develop", type=int, default=1000,
                    help="untimed steps before the warm-up: the droplet oscillates and converts cells every step "
                         "from about step 100 on, so the timed steps see the running regime, not the start")
    ap.add_argument("--impl", default="fsl", choices=["fsl", "reference"])
    ap.add_argument("--workload", default="oscillating256")
    ap.add_argument("--curv", default="lsqr", choices=["lsqr", "fd", "none", "tr"])
    ap.add_argument("--storage", default="f32", choices=["f32", "f16", "bf16"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-side", action="store_true", help="skip the dense-pool and precision-form measurements")
    ap.add_argument("--cpu-seconds", type=float, default=15.0)
    ap.add_argument("--mlp-train", type=int, default=10_000_000, help="training stencils of the learned curvature")
    ap.add_argument("--mlp-epochs", type=int, default=2)
    ap.add_argument("--mlp-batch", type=int, default=4096, help="rows per Adam step of the learned curvature")
    ap.add_argument("--mlp-only", action="store_true",
                    help="run only the MLP training section (no in-step inference) and print it")
    ap.add_argument("--no-physics", action="store_true", help="skip the physics reports of the side sections")
    ap.add_argument("--physics", action="store_true",
                    help="run only the configuration reports (Laplace test, sessile caps, oscillation period)")
    ap.add_argument("--adjoint-only", action="store_true",
                    help="run only the adjoint-window section (one evaluation, no checks) and print it")
    return ap.parse_args()


def dist_info():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


# ---------------------------------------------------------------- clocks
class ClockSampler:
    FIELDS = ("timestamp,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index: int):
        self.rows = []
        try:
            self.proc = subprocess.Popen(["nvidia-smi", f"--query-gpu={self.FIELDS}", "--format=csv,noheader,nounits",
                                          "-lms", "50", "-i", str(index)], stdout=subprocess.PIPE,
                                         stderr=subprocess.DEVNULL, text=True)
        except OSError:
            self.proc = None
            return
        self.t = threading.Thread(target=self._read, daemon=True)
        self.t.start()

    def _read(self):
        for line in self.proc.stdout:
            self.rows.append((time.time(), line.strip()))

    def stop(self):
        if self.proc is None:
            return
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except subprocess.TimeoutExpired:
            self.proc.kill()
        self.t.join(timeout=5)

    def summary(self, t0: float, t1: float) -> dict:
        rows = [(t, r.split(", ")) for t, r in self.rows]
        rows = [(t, r) for t, r in rows if len(r) >= 9]
        inside = [r for t, r in rows if t0 <= t <= t1 + 0.06]
        note = "samples during the timed region"
        if not inside and rows:
            inside = [min(rows, key=lambda tr: min(abs(tr[0] - t0), abs(tr[0] - t1)))[1]]
            note = "timed region shorter than the sampling interval: nearest sample"
        if not inside:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "note": "nvidia-smi unavailable"}

        def num(x):
            try:
                return float(x)
            except ValueError:
                return None

        sm = [num(r[1]) for r in inside if num(r[1]) is not None]
        reasons = set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for r in inside:
            for k, n in enumerate(names):
                if r[5 + k].strip().lower() == "active":
                    reasons.add(n)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": num(inside[0][2]),
                "power_w_max": max((num(r[3]) or 0.0) for r in inside), "reasons": sorted(reasons),
                "samples": len(inside), "note": note}


# ---------------------------------------------------------------- workload
def geometry_kwargs(g: dict) -> dict:
    kw = dict(c=g.get("c", (0, 0, 0)), R=g.get("R", 0.0), eps2=g.get("eps2", 0.0), c2=g.get("c2", (0, 0, 0)),
              R2=g.get("R2", 0.0), zw=g.get("zw", 0.0), h0=g.get("h0", 0.0), amp=g.get("amp", 0.0),
              wavelength=g.get("wavelength", 1.0), sub=16)
    if g["kind"] == "mode2":
        kw["R"] = g["R_s"]
    return kw


def make_sim(F, w, curv, storage, stream):
    import torch
    coll = F.TRT if w["collision"] == "trt" else F.BGK
    cm = {"lsqr": F.CURV_LSQR, "fd": F.CURV_FD, "none": F.CURV_NONE, "tr": F.CURV_TR, "mlp": F.CURV_MLP}[curv]
    st = {"f32": F.F32, "f16": F.F16_OFS, "bf16": F.BF16_OFS}[storage]
    P = F.make_params(w["shape"], collision=coll, curv_model=cm, storage=st, tau=w["tau"], sigma=w["sigma"],
                      theta=w["theta"])
    phi0 = torch.zeros(w["shape"], dtype=torch.float32, device="cuda")
    F.fill_geometry(P, F.make_geometry(w["geometry"]["kind"], **geometry_kwargs(w["geometry"])), phi0, stream)
    obs = None
    if w["walls"]:
        from paper_1509_07691_gb300 import synthetic as S
        obs = torch.from_numpy(S.obstacle_mask(w["shape"], w["walls"])).cuda()
    sim = F.Sim(P, phi0=phi0, obstacle=obs, stream=stream)
    return P, sim, phi0, obs


# ---------------------------------------------------------------- CPU oracle
def oracle_crop(w, z_rows: int | None = None):
    """The workload's droplet cropped to its bounding box (all of its fluid
    cells, gas margin 4) as an FP64 oracle state; with z_rows, only that many
    z rows around the centre (a periodic slab, a bounded sample of the same
    cells).  Returns (params, state, crop shape, fluid cells)."""
    import oracle as orc
    g = w["geometry"]
    R_out = g.get("R_s", g.get("R", 8.0)) * (1 + abs(g.get("eps2", 0.0))) + 1.0
    c = np.array(g["c"])
    lo = np.floor(c - R_out - 4).astype(int)
    hi = np.ceil(c + R_out + 4).astype(int) + 1
    if z_rows is not None and z_rows < hi[2] - lo[2]:
        lo[2] = int(np.floor(c[2])) - z_rows // 2
        hi[2] = lo[2] + z_rows
    ext = hi - lo  # (x, y, z)
    shape = (int(ext[2]), int(ext[1]), int(ext[0]))
    kw = geometry_kwargs(g)
    kw["c"] = tuple(c - lo)
    og = orc.geom(g["kind"], **kw)
    # fill: cells far inside / outside by radial bounds, the band cell by cell with the oracle's sampler
    zz, yy, xx = np.meshgrid(*[np.arange(n) for n in shape], indexing="ij")
    r = np.sqrt((xx - kw["c"][0]) ** 2 + (yy - kw["c"][1]) ** 2 + (zz - kw["c"][2]) ** 2)
    e = abs(kw.get("eps2", 0.0))
    phi = np.where(r + 1.0 < kw["R"] * (1 - 0.5 * e), 1.0, 0.0)
    band = np.nonzero(((r + 1.0 >= kw["R"] * (1 - 0.5 * e)) & (r - 1.0 <= kw["R"] * (1 + e))).ravel())[0]
    phi.ravel()[band] = orc.fill_cells(og, shape, band)
    coll = 1 if w["collision"] == "trt" else 0
    P = orc.params(shape, collision=coll, tau=w["tau"], sigma=w["sigma"], theta=w["theta"], curv_model=0)
    st = orc.init_state(P, phi)
    return P, st, shape, int(np.count_nonzero(st.flags & 3))


def oracle_sample(w, max_seconds: float, gpu_state=None):
    """Time the FP64 oracle on the droplet cropped to its bounding box on one
    host core for about max_seconds; optionally compare the curvature of a GPU
    state with the oracle's on sampled cells."""
    import oracle as orc
    P, st, shape, n_fluid = oracle_crop(w)
    steps, t_used = 0, 0.0
    while t_used < max_seconds and steps < 1000:
        t0 = time.perf_counter()
        st, counts, _, _ = orc.step(P, st)
        t_used += time.perf_counter() - t0
        steps += 1
    out = {"value": n_fluid * steps / t_used / 1e6, "unit": "MLUPS", "cores": 1, "kind": "oracle",
           "sample": f"{steps} FP64 oracle steps (LSQR curvature + step) of the {w['shape'][2]}^3 droplet cropped "
                     f"to its bounding box {shape[2]}x{shape[1]}x{shape[0]} ({n_fluid} fluid cells), single thread",
           "seconds": round(t_used, 3), "steps": steps, "fluid_cells": n_fluid}
    if gpu_state is not None:
        out["kappa_check"] = kappa_error(orc, gpu_state, w)
    return out


def _oracle_rate(args):
    """One process of oracle_all_cores: (fluid cells x steps, stepping seconds)."""
    w, seconds = args
    r = oracle_sample(w, seconds)
    return r["fluid_cells"] * r["steps"], r["seconds"]


def oracle_all_cores(w, seconds: float, processes: int | None = None):
    """The same single-threaded oracle run as oracle_sample, one independent
    process per host core (spawn pool, the oracle itself unchanged): the
    aggregate rate is the sum of the processes' rates over their concurrent
    stepping time."""
    import multiprocessing as mp
    n = processes or os.cpu_count() or 1
    with mp.get_context("spawn").Pool(n) as pool:
        res = pool.map(_oracle_rate, [(w, seconds)] * n)
    rate = sum(u / t for u, t in res if t > 0)
    return {"value": rate / 1e6, "unit": "MLUPS", "cores": n, "kind": "oracle, one process per core",
            "sample": f"{n} processes, each the cpu_baseline sample for about {seconds:g} s of steps"}


def kappa_error(orc, gs, w, n_sample=300, half=3):
    """Oracle LSQR curvature on 7^3 windows (FP32 state cast to FP64) around
    sampled interface cells vs the GPU curvature of the same state."""
    flags, phi, kappa = gs["flags"], gs["phi"], gs["kappa"]
    idx = np.argwhere((flags & 15) == 2)
    pick = idx[(np.linspace(0, len(idx) - 1, min(n_sample, len(idx)))).astype(int)]
    errs, refs = [], []
    P = orc.params((2 * half + 1,) * 3, theta=w["theta"], curv_model=0)
    for z, y, x in pick:
        sl = [np.arange(v - half, v + half + 1) % n for v, n in zip((z, y, x), flags.shape)]
        fw = (flags[np.ix_(*sl)] & 15).astype(np.uint8)
        pw = phi[np.ix_(*sl)].astype(np.float64)
        k, _, _ = orc.curvature(P, fw, pw)
        ref = k[half, half, half]
        refs.append(ref)
        errs.append(abs(kappa[z, y, x] - ref))
    refs, errs = np.array(refs), np.array(errs)
    L = max(flags.shape)
    rel = errs / np.maximum(np.abs(refs), 1.0 / L)
    return {"cells": int(len(pick)), "max_rel": float(rel.max()), "median_rel": float(np.median(rel)),
            "mean_abs_kappa": float(np.mean(np.abs(refs))), "tolerance": 1e-4,
            "definition": "|k_gpu - k_fp64| / max(|k_fp64|, 1/L), FP64 oracle LSQR on the same FP32 fill levels"}


def heldout_errors(held):
    """Relative curvature error of the network and of the FP64 LSQR fit on the
    same noisy held-out droplet stencils (oracle LSQR on each 5^3 stencil)."""
    import oracle as orc
    import oracle.mlp as M
    q, truth, ym = held["params"], held["truth"], held["mlp"]
    P = orc.params((5, 5, 5), curv_model=0)
    kl = []
    for k in range(len(truth)):
        s = M.stencil_fill(q["axes"][k], q["quat"][k], M.shape_centre(q["axes"][k], q["quat"][k], q["dir"][k],
                                                                      q["delta"][k]), 0, 8)
        nz = M.noise_normal(held["noise_seed"], k * 125 + np.arange(125)).reshape(5, 5, 5) * 1e-3
        s = np.where((s > 0) & (s < 1), np.clip(s + nz, 0.0, 1.0), s)
        st = orc.init_state(P, np.transpose(s, (2, 1, 0)).copy())
        kk, _, _ = orc.curvature(P, st.flags, st.phi)
        kl.append(kk[2, 2, 2])
    kl = np.array(kl)
    return {"stencils": int(len(truth)), "radii": "4..48 cells, droplets, noise 1e-3",
            "network_mean_rel": float(np.mean(np.abs(ym - truth) / np.abs(truth))),
            "lsqr_fp64_mean_rel": float(np.mean(np.abs(kl - truth) / np.abs(truth)))}


# ---------------------------------------------------------------- main legs
def run_reference(args):
    """The reference arm: the FP64 oracle as it stands, one host core, on the
    workload's droplet cropped to its bounding box.  Exactly `warmup` untimed
    and `steps` timed oracle steps; if that many steps of the whole crop would
    take more than about REFERENCE_BUDGET_S, each step runs on a z slab of the
    crop instead (the rate is per fluid cell of what was stepped)."""
    ws, rank, _ = dist_info()
    if rank != 0:
        return
    from paper_1509_07691_gb300 import synthetic as S
    import oracle as orc
    w = S.workload(args.workload)
    n_total = max(1, args.steps + args.warmup)
    P, st, shape, n_fluid = oracle_crop(w)
    t0 = time.perf_counter()
    st1, _, _, _ = orc.step(P, st)  # probe step, also the first warm-up step when the crop is kept
    t_probe = time.perf_counter() - t0
    done_warm = 1
    if t_probe * n_total > REFERENCE_BUDGET_S:
        rows = max(8, int(shape[0] * REFERENCE_BUDGET_S / (t_probe * n_total)))
        P, st, shape, n_fluid = oracle_crop(w, z_rows=rows)
        done_warm = 0
        sample = (f"z slab of {shape[0]} rows through the centre of the {w['shape'][2]}^3 droplet's bounding box, "
                  f"{shape[2]}x{shape[1]}x{shape[0]} periodic ({n_fluid} fluid cells)")
    else:
        st = st1
        sample = (f"the {w['shape'][2]}^3 droplet cropped to its bounding box {shape[2]}x{shape[1]}x{shape[0]} "
                  f"({n_fluid} fluid cells)")
    for _ in range(max(0, args.warmup - done_warm)):
        st, _, _, _ = orc.step(P, st)
    t0 = time.perf_counter()
    for _ in range(args.steps):
        st, _, _, _ = orc.step(P, st)
    t_timed = time.perf_counter() - t0
    value = n_fluid * args.steps / max(t_timed, 1e-9) / 1e6
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": "MLUPS", "n_gpus": args.gpus,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * t_timed / max(1, args.steps),
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": f"{args.workload} (cropped to the droplet's bounding box)",
                       "grid": list(w["shape"][::-1]), "timed_from_step": args.warmup,
                       "note": "from the initial droplet: the oracle's time per fluid-cell update does not depend "
                               "on how far the droplet has developed"},
            "cpu_baseline": {"value": value, "unit": "MLUPS", "cores": 1, "kind": "oracle",
                             "sample": f"{args.warmup} untimed + {args.steps} timed FP64 oracle steps (LSQR curvature "
                                       f"+ step) of {sample}, single thread"},
            "e2e": {"value": value, "unit": "MLUPS", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


REFERENCE_BUDGET_S = 120.0

PHASES = ["normals_plic", "lsqr_curvature", "sc_liquid", "sc_interface", "convert", "finalize"]


def algorithmic_bytes(n_fluid, n_if, n_seg_cells, fused=False, pdf_bytes=4):
    """Bytes each phase must move at least, per launch.  Per interface cell:
    normals 21 B (phi and flag read, normal and offset written), LSQR fit 21 B
    (normal and flag read, kappa written), interface stream-collide 57 PDFs
    (own 19 read, 18 pulled, 19 written) plus m, phi, kappa, rho and the flag
    (20 B); per liquid cell 38 PDFs plus 1 B of flags per segment cell; the
    final update 14 B per interface cell.  fused: the LSQR fit and the
    interface stream-collide run as one pass (phase lsqr_curvature; the
    sc_interface phase holds the deferred cells).  pdf_bytes: 4 for FP32
    PDFs, 2 for the 16-bit offset forms."""
    nb = {"normals_plic": 21.0 * n_if,           # phi + flag read, normal + offset written
          "lsqr_curvature": 21.0 * n_if,         # normal + flag read, kappa written
          "sc_liquid": 38.0 * pdf_bytes * (n_fluid - n_if) + 1.0 * n_seg_cells,  # 19 PDFs in + 19 out, flags
          "sc_interface": (57.0 * pdf_bytes + 20.0) * n_if,  # own + pulled + written PDFs, m, phi, kappa, rho, flag
          "convert": 0.0, "finalize": 14.0 * n_if}
    if fused:
        nb["lsqr_curvature"] += nb["sc_interface"]
        nb["sc_interface"] = 0.0
    return nb


def time_steps(sim, steps, stream, flush):
    import torch
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
    for k in range(steps):
        flush.fill_(float(k))
        ev[k][0].record(stream)
        sim.step(1)
        ev[k][1].record(stream)
    torch.cuda.synchronize()
    return sum(a.elapsed_time(b) for a, b in ev)


def phase_profile(sim, nprof, flush):
    ph = np.zeros(len(PHASES))
    for k in range(nprof):
        flush.fill_(float(k))
        ph += sim.step_profile()
    return ph / nprof


def launches_per_step(curv, obs):
    """Kernels of one recorded step: normals, the curvature (LSQR: the fused fit
    + interface stream-collide, plus the general-path kernel when some cell has
    an obstacle neighbour; FD / none: curvature, then the interface
    stream-collide), the liquid stream-collide, conversion and the two final
    updates."""
    if curv == "lsqr":
        return 7 if obs is not None and bool(obs.any()) else 6
    return 7


def kernels_per_step(curv, obs):
    """The same less the normals, which FD curvature leaves out in a domain
    without obstacles."""
    return launches_per_step(curv, obs) - (1 if curv == "fd" and (obs is None or not bool(obs.any())) else 0)


def measured_traffic(kernel, workload):
    """DRAM bytes per launch from the committed ncu capture (profiles/ncu_traffic.json),
    or None when the kernel's source changed since the capture."""
    import hashlib
    try:
        data = json.load(open(os.path.join(ROOT, "profiles", "ncu_traffic.json")))
    except (OSError, ValueError):
        return None
    for e in data.get("entries", []):
        if e["kernel"] != kernel or e["workload"] != workload:
            continue
        h = hashlib.sha256()
        for f in e["source_files"]:
            h.update(open(os.path.join(ROOT, "paper_1509_07691_gb300", "csrc", f), "rb").read())
        return float(e["bytes_per_launch"]) if h.hexdigest()[:16] == e["source_sha"] else None
    return None


def roofline_of(ph, nbytes, peaks, which=None, workload=None, fused=False):
    k = which if which is not None else int(np.argmax(ph))
    name = PHASES[k]
    label = "lsqr_curvature+sc_interface (fused)" if fused and name == "lsqr_curvature" else name
    hbm = peaks.get("hbm_gbs", 6800.0)
    ach = nbytes[name] / (ph[k] * 1e-3) / 1e9
    return {"kernel": label, "bound": "hbm", "unit": "GB/s", "achieved": ach, "peak": hbm, "frac": ach / hbm,
            "peak_source": "MEASURED_PEAKS.json hbm_gbs (copy, burst; of measured)" if peaks else "fallback 6.8 TB/s",
            "traffic": measured_traffic(name, workload) if workload else None,
            "traffic_source": "profiles/ncu_traffic.json (ncu dram bytes per launch)",
            "algorithmic_bytes": nbytes[name], "launch_ms": float(ph[k])}


def side_workload(F, S, name, storage, steps, stream, flush, peaks, seed):
    """MLUPS and the liquid stream-collide roofline of one more workload."""
    import torch
    w = S.workload(name, seed=seed)
    P, sim, phi0, obs = make_sim(F, w, "lsqr", storage, stream)
    sim.step(5)
    torch.cuda.synchronize()
    st = sim.stats()
    n_fluid, n_if = int(st[0] + st[1]), int(st[1])
    m0, l0 = sim.mass_total()
    ms = time_steps(sim, steps, stream, flush)
    m1, l1 = sim.mass_total()
    ph = phase_profile(sim, min(steps, 20), flush)
    nseg_cells = n_fluid  # liquid rows are dense in this workload
    nb = algorithmic_bytes(n_fluid, n_if, nseg_cells, fused=True, pdf_bytes=4 if storage == "f32" else 2)
    out = {"workload": name, "storage": storage, "fluid_cells": n_fluid, "interface_cells": n_if,
           "mlups": n_fluid * steps / (ms * 1e-3) / 1e6, "ms_per_step": ms / steps,
           "mass_drift_rel": ((m1 + l1) - (m0 + l0)) / (m0 + l0), "mass_drift_steps": steps,
           "phases_ms": dict(zip(PHASES, [round(float(v), 5) for v in ph])),
           "roofline_sc_liquid": roofline_of(ph, nb, peaks, which=PHASES.index("sc_liquid"),
                                             workload=name if storage == "f32" else None)}
    sim.close()
    del sim, phi0, obs
    torch.cuda.empty_cache()
    return out


def learned_curvature(F, S, stream, flush, peaks, seed, n_train, epochs, steps, inference=True, batch=4096):
    """Config-5 form: train the network on GPU-made stencils, then run the
    384^3 two-droplet coalescence with FSL_CURV_MLP (LSQR judge, 5 %)."""
    import torch
    out = {}
    p = S.mlp_sample_params(seed, n_train)
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    X, target = F.mlp_stencils(p, sub=8, noise=1e-3, noise_seed=seed + 1)
    torch.cuda.synchronize()
    gen_s = time.perf_counter() - t0
    net = F.Mlp(S.mlp_init_weights(seed + 2))
    B = batch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    losses = torch.zeros(n_train // B, dtype=torch.float32, device="cuda")
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    nsteps = 0
    for ep in range(epochs):
        perm = torch.randperm(n_train, device="cuda", generator=gen)
        lr = 2e-3 * (0.5 ** ep)
        nsteps += net.train_epoch(X, target, perm, B, lr, losses=losses)  # batch loop in the library
    torch.cuda.synchronize()
    train_s = time.perf_counter() - t0
    out["training"] = {"stencils": n_train, "sub_samples": 8, "noise": 1e-3, "stencils_per_s": n_train / gen_s,
                       "epochs": epochs, "batch": B, "steps": nsteps, "samples_per_s": nsteps * B / train_s,
                       "final_batch_loss": float(losses[-1].item()),
                       "last_epoch_mean_loss": float(losses.double().mean().item()),
                       "loop": "fsl_mlp_train_epoch: per batch one fused tensor-core tile kernel (rows gathered by the permutation) and one reduction + Adam kernel, one C-ABI call per epoch",
                       "flops_per_sample": 3 * 2 * (128 * 128 * 2 + 128)}
    del X, target
    torch.cuda.empty_cache()
    # held-out stencils for the kappa error (network here; LSQR in the CPU leg)
    nt = 256
    q = S.mlp_sample_params(seed + 3, nt)
    R = np.exp(np.log(4.0) + S.uniform(seed + 4, nt) * (np.log(48.0) - np.log(4.0)))
    q["axes"] = np.stack([R, R, R], 1)
    q["invert"] = np.zeros(nt, np.int32)
    Xt, tt = F.mlp_stencils(q, sub=8, noise=1e-3, noise_seed=seed + 5)
    yt = net.forward(Xt).cpu().numpy()
    out["heldout"] = {"params": q, "noise_seed": seed + 5, "truth": tt.cpu().numpy(), "mlp": yt}
    out["net"] = net
    if not inference:
        return out
    # inference inside FSLBM
    w = S.workload("coalescence384", seed=seed)
    P = F.make_params(w["shape"], collision=F.BGK, curv_model=F.CURV_MLP, tau=w["tau"], sigma=w["sigma"],
                      theta=w["theta"])
    phi0 = torch.zeros(w["shape"], dtype=torch.float32, device="cuda")
    F.fill_geometry(P, F.make_geometry(w["geometry"]["kind"], **geometry_kwargs(w["geometry"])), phi0, stream)
    sim = F.Sim(P, phi0=phi0, stream=stream)
    sim.attach_mlp(net, 0.05)
    sim.step(5)
    torch.cuda.synchronize()
    st = sim.stats()
    n_fluid, n_if = int(st[0] + st[1]), int(st[1])
    ms = time_steps(sim, steps, stream, flush)
    st = sim.stats()
    kap = torch.empty_like(sim.kappa)
    cev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(10)]
    for a, b in cev:
        flush.fill_(1.0)
        a.record(stream)
        sim.curvature(F.CURV_MLP, kap)
        b.record(stream)
    torch.cuda.synchronize()
    cm = sum(a.elapsed_time(b) for a, b in cev) / len(cev)
    for a, b in cev:  # the LSQR part alone on the same state: the network's share is the difference
        flush.fill_(1.0)
        a.record(stream)
        sim.curvature(F.CURV_LSQR, kap)
        b.record(stream)
    torch.cuda.synchronize()
    cl = sum(a.elapsed_time(b) for a, b in cev) / len(cev)
    out["inference"] = {"workload": "coalescence384", "grid": list(w["shape"][::-1]), "fluid_cells": n_fluid,
                        "interface_cells": n_if, "mlups": n_fluid * steps / (ms * 1e-3) / 1e6, "ms_per_step": ms / steps,
                        "mlp_cells_last_step": int(st[8]), "kept_fraction": float(st[9]) / max(1, int(st[8])),
                        "curvature_ms_lsqr_plus_mlp": cm, "curvature_ms_lsqr": cl,
                        "network_ms": cm - cl, "network_flops_per_s": n_if * 2 * (125 * 128 + 128 * 128 + 128) / ((cm - cl) * 1e-3),
                        "curvature_evals_per_s": n_if / (cm * 1e-3)}
    sim.close()
    del sim, phi0
    torch.cuda.empty_cache()
    return out


def adjoint_window(F, S, stream, seed, window=50, ckpt=10, reps=5, warm=2, checks=True):
    """Differentiation form: sessile droplet 64^3 (R 16, walls), windows of 50
    steps with frozen cell types and a checkpoint every 10 steps.  Loss: L2 of
    the interface fill levels against the window run at theta 70 deg, sigma
    3e-4; gradient at theta 90 deg, sigma 2e-4 by the reverse pass; timing of
    the forward window and of the reverse pass; L-BFGS fit through the
    autograd Function from the start point."""
    import torch
    from scipy.optimize import minimize
    w = S.workload("sessile64", seed=seed)
    P, sim, phi0, obs = make_sim(F, w, "lsqr", "f32", stream)
    start = sim.snapshot()
    sim.curvature(F.CURV_LSQR, torch.empty_like(sim.kappa))
    fp64_cells = int(sim.stats()[6])
    th0, s0 = math.radians(90.0), 2e-4
    th1, s1 = math.radians(70.0), 3e-4
    sim.set_surface(s1, th1)
    sim.window_forward(window, ckpt)
    torch.cuda.synchronize()
    tgt = sim.phi.clone()
    ifc = (sim.flags_current() & F.TYPE_MASK) == F.INTERFACE
    n_if = int(ifc.sum())
    n_fluid = int(((sim.flags_current() & F.TYPE_MASK) & (F.LIQUID | F.INTERFACE) != 0).sum())
    e = [torch.cuda.Event(enable_timing=True) for _ in range(3)]

    def evaluate(theta, sigma, grad=False):
        sim.restore(start)
        sim.set_surface(sigma, theta)
        e[0].record(stream)
        sim.window_forward(window, ckpt)
        e[1].record(stream)
        d = torch.where(ifc, sim.phi - tgt, torch.zeros_like(tgt))
        L = float(torch.sum(d.double() ** 2))
        if not grad:
            return L, e[0].elapsed_time(e[1])
        g = 2.0 * d
        torch.cuda.synchronize()
        e[1].record(stream)
        ds, dt = sim.window_adjoint(g)
        e[2].record(stream)
        torch.cuda.synchronize()
        return L, ds, dt, e[0].elapsed_time(e[1]), e[1].elapsed_time(e[2])

    for _ in range(warm):
        evaluate(th0, s0, grad=True)
    fwd, bwd = [], []
    for _ in range(reps):
        L, ds, dt, tf, tb = evaluate(th0, s0, grad=True)
        fwd.append(tf)
        bwd.append(tb)
    tfw, tbw = float(np.median(fwd)), float(np.median(bwd))
    out = {"workload": "sessile64", "grid": list(w["shape"][::-1]), "window": window, "checkpoint_every": ckpt,
           "fluid_cells": n_fluid, "interface_cells": n_if, "lsqr_fp64_cells_at_start": fp64_cells,
           "target": {"theta_deg": 70.0, "sigma": s1},
           "start": {"theta_deg": 90.0, "sigma": s0}, "loss": L, "dL_dsigma": ds, "dL_dtheta": dt,
           "forward_ms": tfw, "reverse_ms": tbw, "reverse_over_forward": tbw / tfw,
           "forward_mlups": n_fluid * window / (tfw * 1e-3) / 1e6,
           "reverse_mlups": n_fluid * window / (tbw * 1e-3) / 1e6}
    if not checks:
        sim.close()
        return out
    hs, ht = 5e-2 * s0, 1e-2
    fd_s = (evaluate(th0, s0 + hs)[0] - evaluate(th0, s0 - hs)[0]) / (2 * hs)
    fd_t = (evaluate(th0 + ht, s0)[0] - evaluate(th0 - ht, s0)[0]) / (2 * ht)
    scale = np.array([1e-4, math.radians(10.0)])
    nev = [0]

    def fun(xs):
        surface = torch.tensor(xs * scale, dtype=torch.float64, requires_grad=True)
        sim.restore(start)
        phi = F.FslStepWindow.apply(surface, sim, window, ckpt)
        loss = torch.sum(torch.where(ifc, phi - tgt, torch.zeros_like(tgt)).double() ** 2)
        loss.backward()
        nev[0] += 1
        return float(loss.detach()), surface.grad.numpy() * scale

    t0 = time.perf_counter()
    res = minimize(fun, np.array([s0, th0]) / scale, jac=True, method="L-BFGS-B", bounds=[(0.5, 6.0), (3.0, 15.0)],
                   options=dict(maxiter=60, ftol=1e-14, gtol=1e-12))
    fit_s = time.perf_counter() - t0
    sf, tf_ = res.x * scale
    out.update({"fp32_differences": {"dL_dsigma": fd_s, "dL_dtheta": fd_t, "step_sigma": hs, "step_theta_rad": ht,
                                "rel_err_sigma": abs(ds - fd_s) / abs(fd_s), "rel_err_theta": abs(dt - fd_t) / abs(fd_t)},
           "fit": {"theta_deg": math.degrees(tf_), "sigma": sf, "theta_err_deg": math.degrees(tf_) - 70.0,
                   "sigma_rel_err": sf / s1 - 1.0, "evaluations": nev[0], "seconds": fit_s,
                   "method": "L-BFGS-B on (sigma/1e-4, theta/10 deg), gradients from the reverse pass"}})
    sim.close()
    del sim, phi0, obs, start
    torch.cuda.empty_cache()
    return out


def _oracle_window_loss(args):
    """One FP64 oracle window (frozen types) of the sessile droplet; returns
    phi at its end, or the L2 loss to `target` on interface cells."""
    name, theta, sigma, window, target = args
    import oracle as orc
    from paper_1509_07691_gb300 import synthetic as S
    w = S.workload(name)
    g = w["geometry"]
    phi = orc.fill(orc.geom("cap", c=g["c"], R=g["R"], zw=g["zw"], sub=16), w["shape"])
    obs = S.obstacle_mask(w["shape"], w["walls"])
    P = orc.params(w["shape"], collision=1, tau=w["tau"], sigma=sigma, theta=theta, frozen=1)
    st = orc.init_state(P, phi, obs)
    for _ in range(window):
        st, _, _, _ = orc.step(P, st)
    if target is None:
        return st.phi, st.flags
    m = st.flags == 2
    return float(np.sum((st.phi[m] - target[m]) ** 2))


def adjoint_reference(window=50):
    """FP64 reference gradient of the adjoint section's loss: central
    differences (h = 1e-4 relative) of the oracle's frozen-type window, the
    target made by the oracle itself; windows run in a spawn pool."""
    import multiprocessing as mp
    th0, s0 = math.radians(90.0), 2e-4
    t0 = time.perf_counter()
    ctx = mp.get_context("spawn")
    with ctx.Pool(1) as pool:
        target, _ = pool.apply(_oracle_window_loss, (("sessile64", math.radians(70.0), 3e-4, window, None),))
    hs, ht = 1e-4 * s0, 1e-4
    jobs = [("sessile64", th0, s0 + hs, window, target), ("sessile64", th0, s0 - hs, window, target),
            ("sessile64", th0 + ht, s0, window, target), ("sessile64", th0 - ht, s0, window, target)]
    with ctx.Pool(4) as pool:
        Ls = pool.map(_oracle_window_loss, jobs)
    return {"dL_dsigma": (Ls[0] - Ls[1]) / (2 * hs), "dL_dtheta": (Ls[2] - Ls[3]) / (2 * ht), "step_sigma": hs,
            "step_theta_rad": ht, "seconds": time.perf_counter() - t0, "processes": 4,
            "method": "central differences of the FP64 oracle window (frozen types), own target"}


def _fill_weight(F, sim):
    """Liquid fraction per cell: 1 in liquid, phi in interface, 0 elsewhere (device tensor)."""
    import torch
    fl = sim.flags_current() & F.TYPE_MASK
    one = torch.ones_like(sim.phi)
    return torch.where(fl == F.LIQUID, one, torch.where(fl == F.INTERFACE, sim.phi, torch.zeros_like(one)))


def zero_crossings(a, every):
    """Times of the sign changes of samples a[k] taken at t = k * every, by
    linear interpolation between the two samples around each change."""
    a = np.asarray(a, dtype=np.float64)
    t = np.arange(len(a)) * every
    return [float(t[i] + every * a[i] / (a[i] - a[i + 1])) for i in range(len(a) - 1) if a[i] * a[i + 1] < 0]


def _velocity(F, sim):
    """(rho, u[3]) of the current PDFs (device tensors)."""
    import torch
    f = sim.pdfs_float()
    c = torch.tensor([[0, 1, -1, 0, 0, 0, 0, 1, -1, 1, -1, 1, -1, 1, -1, 0, 0, 0, 0],
                      [0, 0, 0, 1, -1, 0, 0, 1, -1, -1, 1, 0, 0, 0, 0, 1, -1, 1, -1],
                      [0, 0, 0, 0, 0, 1, -1, 0, 0, 0, 0, 1, -1, -1, 1, 1, -1, -1, 1]],
                     dtype=torch.float32, device=f.device)
    rho = f.sum(0)
    return rho, torch.einsum("dq,qzyx->dzyx", c, f) / rho


def laplace_report(F, S, stream, curv, storage, net=None):
    """Static droplet (droplet32: 32^3, R = 8, sigma = 1e-4, tau = 1, 200
    steps): max spurious |u| over the fluid cells, the Laplace pressure
    (rho_core - 3 p_g)/3 against 2 sigma/R (R from the liquid volume, core =
    liquid cells within R/2 of the centre), the curvature of the interface
    cells against 1/R (mean of kappa R and its r.m.s. deviation from 1) and
    the mass drift."""
    import torch
    w = S.workload("droplet32")
    P, sim, phi0, obs = make_sim(F, w, curv, storage, stream)
    if curv == "mlp":
        sim.attach_mlp(net, 0.05)
    m0, l0 = sim.mass_total()
    sim.step(w["steps"])
    m1, l1 = sim.mass_total()
    rho, u = _velocity(F, sim)
    fl = sim.flags_current() & F.TYPE_MASK
    fluid = (fl == F.LIQUID) | (fl == F.INTERFACE)
    umag = torch.sqrt((u * u).sum(0))[fluid]
    wgt = _fill_weight(F, sim)
    R = (3.0 * float(wgt.sum()) / (4.0 * math.pi)) ** (1.0 / 3.0)
    g = w["geometry"]["c"]
    zz, yy, xx = torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.float32) for n in w["shape"]],
                                indexing="ij")
    r = torch.sqrt((xx - g[0]) ** 2 + (yy - g[1]) ** 2 + (zz - g[2]) ** 2)
    core = (fl == F.LIQUID) & (r < 0.5 * R)
    dp = (float(rho[core].mean()) - 3.0 * P.p_gas) / 3.0
    kap = torch.empty_like(sim.kappa)
    cm = {"lsqr": F.CURV_LSQR, "fd": F.CURV_FD, "tr": F.CURV_TR, "mlp": F.CURV_MLP}[curv]
    sim.curvature(cm, kap)
    kr = kap[fl == F.INTERFACE].double() * R
    out = {"max_u": float(umag.max()), "mean_u": float(umag.mean()), "dp": dp, "dp_laplace": 2.0 * w["sigma"] / R,
           "R_volume": R, "dp_rel_err": abs(dp - 2.0 * w["sigma"] / R) / (2.0 * w["sigma"] / R),
           "kappa_R_mean": float(kr.mean()), "kappa_R_rms_err": float(torch.sqrt(((kr - 1.0) ** 2).mean())),
           "mass_drift_rel": ((m1 + l1) - (m0 + l0)) / (m0 + l0), "steps": w["steps"], "storage": storage}
    if curv == "mlp":
        st = sim.stats()
        out["mlp_kept_fraction"] = float(st[9]) / max(1, int(st[8]))
    sim.close()
    return out


# steps of the sessile caps: the configuration's 5000 steps and on to near equilibrium
CAP_RELAX_STEPS = 60000

# Tab. advection as printed (percent): d -> (L1, L2) for convective and diffusive scaling
ADVECTION_TABLE = {10: ((3.00, 9.38), (3.00, 9.38)), 20: ((1.63, 7.19), (1.38, 6.17)),
                   40: ((1.25, 7.38), (0.85, 5.39)), 80: ((1.17, 8.44), (0.68, 5.87))}


def advection_report(F, stream, diameters=(10, 20, 40, 80)):
    """Tab. advection (Sec. III.A): a gas bubble of diameter d in a periodic
    box of 2d cells carried by a prescribed constant flow (f = feq(1, u0)
    before every step, fsl_prescribe_flow) for T = d/u0 steps; L1 and L2 of
    the bubble indicator 1 - phi against the initial field shifted by d (the
    domain-independent reading of the paper's norms).  Convective scaling:
    u0 = 0.05; diffusive: u0 = 0.05 * 10 / d."""
    import torch
    out = {}
    for d in diameters:
        row = {}
        for k, (name, u0) in enumerate((("convective", 0.05), ("diffusive", 0.05 * 10.0 / d))):
            L = 2 * d
            shape = (L, L, L)
            P = F.make_params(shape, tau=1.0, sigma=0.0, curv_model=F.CURV_NONE)
            phi0 = torch.zeros(shape, dtype=torch.float32, device="cuda")
            F.fill_geometry(P, F.make_geometry("sphere", c=(L / 2, L / 2, L / 2), R=d / 2.0, invert=1, sub=16), phi0,
                            stream)
            sim = F.Sim(P, phi0=phi0, stream=stream)
            g0 = 1.0 - sim.phi.double()
            T = int(round(d / u0))
            t0 = time.perf_counter()
            for _ in range(T):
                sim.prescribe_flow(1.0, (u0, 0.0, 0.0))
                sim.step(1)
            torch.cuda.synchronize()
            sec = time.perf_counter() - t0
            g1 = 1.0 - torch.roll(sim.phi.double(), -d, dims=2)
            l1 = float((g1 - g0).abs().sum() / g0.sum())
            l2 = float(torch.sqrt(((g1 - g0) ** 2).sum() / (g0 ** 2).sum()))
            p1, p2 = ADVECTION_TABLE.get(d, ((None, None), (None, None)))[k]
            row[name] = {"u0": u0, "steps": T, "L1_pct": 100 * l1, "L2_pct": 100 * l2, "paper_L1_pct": p1,
                         "paper_L2_pct": p2, "seconds": sec}
            sim.close()
        out[str(d)] = row
    return out


def renardy_bubble(F, stream, dx_inv, curv, steps, moving=False, sample_every=0):
    """The Laplace test of Sec. III.A on a bubble (Renardy's setup): unit box,
    R = 0.125, rho = 4, mu = 1, sigma = 0.357, gas pressure by the bubble
    model.  Lattice units at dx = 1/dx_inv under the paper's time steps
    (dt = 1e-4 (48/dx_inv)^2): nu = mu/rho dt/dx^2, tau = 3 nu + 1/2,
    sigma_lb = sigma/rho dt^2/dx^3, R = dx_inv/8 cells.  Static frame: no-slip
    walls at z = 0 and 1 (obstacle layers), periodic in x and y.  Moving frame
    (moving=True): u0 = 0.0024 along x added to the liquid, periodic in all
    directions (reading E2: a background flow with no-slip walls would be
    sheared), run for T = L/u0 steps.  Reports the maximum spurious |u| (in
    the moving frame |u - u0|) over fluid cells, in lattice units and in
    units of the box per unit time (x dx/dt), and L2(kappa) = sqrt(sum
    (kappa + 1/R)^2 / sum (1/R)^2) over the interface cells."""
    import torch
    L = dx_inv
    dt = 1e-4 * (48.0 / dx_inv) ** 2
    dx = 1.0 / dx_inv
    nu = 0.25 * dt / dx ** 2
    tau = 3.0 * nu + 0.5
    sig = 0.357 / 4.0 * dt ** 2 / dx ** 3
    R = L / 8.0
    u0 = 0.0024 if moving else 0.0
    if moving:
        shape, walls = (L, L, L), None
        c = (L / 2 + 0.13, L / 2 - 0.21, L / 2 + 0.07)
    else:
        shape = (L + 2, L, L)
        walls = torch.zeros(shape, dtype=torch.uint8, device="cuda")
        walls[0] = 1
        walls[-1] = 1
        c = (L / 2 + 0.13, L / 2 - 0.21, (L + 2) / 2 - 0.5 + 0.07)
    cm = {"lsqr": F.CURV_LSQR, "fd": F.CURV_FD, "tr": F.CURV_TR}[curv]
    P = F.make_params(shape, tau=tau, sigma=sig, curv_model=cm)
    phi0 = torch.zeros(shape, dtype=torch.float32, device="cuda")
    F.fill_geometry(P, F.make_geometry("sphere", c=c, R=R, invert=1, sub=16), phi0, stream)
    if walls is not None:
        phi0[walls > 0] = 0.0
    sim = F.Sim(P, phi0=phi0, obstacle=walls, stream=stream)
    if moving:
        sim.prescribe_flow(1.0, (u0, 0.0, 0.0))  # initial liquid state: feq(1, u0)
    sim.set_bubble(1.0 / 3.0)
    hist = []

    def l2k():
        kap = torch.empty_like(sim.kappa)
        sim.curvature(cm, kap)
        fl = sim.flags_current() & F.TYPE_MASK
        k = kap[fl == F.INTERFACE].double()
        return float(torch.sqrt(((k + 1.0 / R) ** 2).sum() / (k.numel() / R ** 2)))

    done = 0
    t0 = time.perf_counter()
    while done < steps:
        n = min(steps - done, sample_every or steps)
        sim.step(n)
        done += n
        if sample_every:
            hist.append((done, l2k()))
    torch.cuda.synchronize()
    sec = time.perf_counter() - t0
    rho, u = _velocity(F, sim)
    fl = sim.flags_current() & F.TYPE_MASK
    fluid = (fl == F.LIQUID) | (fl == F.INTERFACE)
    u[0] -= u0
    umag = torch.sqrt((u * u).sum(0))[fluid]
    out = {"dx": dx, "dt": dt, "tau": tau, "sigma_lb": sig, "R_cells": R, "grid": list(shape[::-1]), "steps": steps,
           "max_u_lb": float(umag.max()), "mean_u_lb": float(umag.mean()),
           "max_u_box_units": float(umag.max()) * dx / dt, "L2_kappa": l2k(), "bubble": list(sim.bubble()),
           "seconds": sec}
    if hist:
        out["L2_kappa_history"] = hist
    sim.close()
    return out


def physics_reports(F, S, stream, net=None):
    """The quantities the workload configurations ask to report, measured on the
    GPU path with plain torch reductions of the state (diagnostics, not the hot
    path):
      droplet32 (200 steps): laplace_report for the LSQR, FD and TR models in
        FP32, LSQR with FP16 and BF16 offset storage, and the learned
        curvature (LSQR judge) when a trained network is given;
      sessile128 (theta = 30, 60, 90, 120 deg): apex height and contact radius
        of the cap against the spherical cap of the conserved volume at that
        angle after CAP_RELAX_STEPS steps (the height after the configuration's
        5000 steps beside it);
      oscillating256 (36000 steps, about two periods), FP32 and the FP16 and
        BF16 offset forms: mode-2 period from the zero crossings of the
        quadrupole moment against Rayleigh's inviscid value and Lamb's damped
        one, and the mass drift;
      full256 (256^3, every cell liquid, at rest): the liquid stream-collide
        alone against the copy bandwidth."""
    import torch
    out = {}
    lap = {}
    for key, curv, storage in (("lsqr", "lsqr", "f32"), ("fd", "fd", "f32"), ("tr", "tr", "f32"),
                               ("lsqr_f16", "lsqr", "f16"), ("lsqr_bf16", "lsqr", "bf16")):
        lap[key] = laplace_report(F, S, stream, curv, storage)
    if net is not None:
        lap["mlp"] = laplace_report(F, S, stream, "mlp", "f32", net)
    out["laplace_droplet32"] = lap
    # -- sessile caps
    caps = {}
    for th in (30.0, 60.0, 90.0, 120.0):
        w = S.workload("sessile128", theta_deg=th)
        P, sim, phi0, obs = make_sim(F, w, "lsqr", "f32", stream)
        vol0 = float(_fill_weight(F, sim).sum())
        sim.step(w["steps"])
        early = {"height": float(_fill_weight(F, sim).sum(0).max()), "steps": w["steps"]}
        sim.step(CAP_RELAX_STEPS - w["steps"])  # the spreading takes many capillary-viscous times
        wgt = _fill_weight(F, sim)
        vol = float(wgt.sum())
        h = float(wgt.sum(0).max())  # apex column: cells above the wall layer z = 0
        r_wet = math.sqrt(float(wgt[1].sum()) / math.pi)  # footprint in the first layer above the wall
        ct, st_ = math.cos(math.radians(th)), math.sin(math.radians(th))
        Rc = (3.0 * vol / (math.pi * (1.0 - ct) ** 2 * (2.0 + ct))) ** (1.0 / 3.0)
        h_cap, r_cap = Rc * (1.0 - ct), Rc * st_
        caps[f"{th:g}"] = {"height": h, "height_cap": h_cap, "rel_err": abs(h - h_cap) / h_cap,
                           "contact_radius": r_wet, "contact_radius_cap": r_cap,
                           "contact_radius_rel_err": abs(r_wet - r_cap) / r_cap,
                           "volume": vol, "volume_drift_rel": (vol - vol0) / vol0, "steps": CAP_RELAX_STEPS,
                           "at_config_steps": early}
        sim.close()
    out["sessile128_caps"] = caps
    # -- oscillation period, per storage form
    per_all = {}
    for storage in ("f32", "f16", "bf16"):
        w = S.workload("oscillating256")
        P, sim, phi0, obs = make_sim(F, w, "lsqr", storage, stream)
        zz, yy, xx = torch.meshgrid(*[torch.arange(n, device="cuda", dtype=torch.float32) for n in w["shape"]],
                                    indexing="ij")
        every, total = 200, 36000
        a = []
        m0, l0 = sim.mass_total()
        for k in range(total // every + 1):
            if k:
                sim.step(every)
            wgt = _fill_weight(F, sim)
            m = wgt.sum()
            cx, cy, cz = (wgt * xx).sum() / m, (wgt * yy).sum() / m, (wgt * zz).sum() / m
            izz = (wgt * (zz - cz) ** 2).sum() / m
            ixy = 0.5 * ((wgt * (xx - cx) ** 2).sum() + (wgt * (yy - cy) ** 2).sum()) / m
            a.append(float(izz - ixy))
        m1, l1 = sim.mass_total()
        sim.close()
        del xx, yy, zz
        zc = zero_crossings(a, every)
        R = w["geometry"]["R"]
        nu = (w["tau"] - 0.5) / 3.0
        w0 = math.sqrt(8.0 * w["sigma"] / R ** 3)  # l (l - 1) (l + 2) = 8 for l = 2, rho = 1
        gam = 5.0 * nu / R ** 2                      # (l - 1)(2 l + 1) nu / R^2
        per = {"zero_crossings": [float(v) for v in zc], "samples_every": every, "steps": total,
               "period_rayleigh": 2.0 * math.pi / w0,
               "period_lamb_damped": 2.0 * math.pi / math.sqrt(max(w0 * w0 - gam * gam, 1e-30)),
               "mass_drift_rel": ((m1 + l1) - (m0 + l0)) / (m0 + l0), "amplitude_first": a[0], "amplitude_last": a[-1]}
        if len(zc) >= 2:
            per["period"] = 2.0 * float(np.mean(np.diff(zc)))
            per["rel_err_lamb"] = abs(per["period"] - per["period_lamb_damped"]) / per["period_lamb_damped"]
        per_all[storage] = per
        torch.cuda.empty_cache()
    out["oscillating256_period"] = per_all
    # -- Tab. advection (prescribed flow)
    out["advection_table"] = advection_report(F, stream)
    # -- Renardy bubble with the bubble model: static (short run) and moving frame
    out["renardy_static_dx48"] = {m: renardy_bubble(F, stream, 48, m, 20000) for m in ("fd", "lsqr", "tr")}
    out["renardy_moving_dx96"] = {m: renardy_bubble(F, stream, 96, m, 40000, moving=True, sample_every=4000)
                                  for m in ("fd", "lsqr", "tr")}
    # -- all-liquid box: the liquid stream-collide alone
    shape = (256, 256, 256)
    P = F.make_params(shape, collision=F.BGK, tau=0.6)
    sim = F.Sim(P, phi0=torch.ones(shape, dtype=torch.float32, device="cuda"), stream=stream)
    sim.step(5)
    ms = time_steps(sim, 50, stream, torch.empty(64 << 20, dtype=torch.float32, device="cuda"))
    n = shape[0] * shape[1] * shape[2]
    gbs = 152.0 * n / (ms / 50 * 1e-3) / 1e9
    out["full256"] = {"ms_per_step": ms / 50, "mlups": n / (ms / 50 * 1e-3) / 1e6, "achieved_gbs": gbs,
                      "bytes_per_cell": 152, "note": "at rest (f = w_q); the step is the liquid stream-collide plus "
                                                     "the empty list kernels"}
    sim.close()
    return out


def reduce_over_ranks(ms, n_fluid, device):
    """Timed milliseconds (max over ranks) and fluid cells (sum over ranks) of
    the default process group; the values themselves on a single process."""
    import torch
    import torch.distributed as dist
    if not (dist.is_available() and dist.is_initialized()) or dist.get_world_size() == 1:
        return float(ms), float(n_fluid)
    t = torch.tensor([ms], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    n = torch.tensor([n_fluid], dtype=torch.float64, device=device)
    dist.all_reduce(n)
    return float(t.item()), float(n.item())


def run_fsl(args):
    import torch
    ws, rank, local = dist_info()
    if ws > 1:
        import torch.distributed as dist
        os.environ.setdefault("MASTER_ADDR", "127.0.0.1")
        dist.init_process_group("nccl" if torch.cuda.is_available() else "gloo")
    torch.cuda.set_device(local)
    from paper_1509_07691_gb300 import build as B
    B.build()
    from paper_1509_07691_gb300 import fsl as F
    from paper_1509_07691_gb300 import synthetic as S
    peaks = {}
    try:
        peaks = json.load(open(os.path.join(ROOT, "MEASURED_PEAKS.json")))
    except OSError:
        pass
    w = S.workload(args.workload, seed=S.SEED + rank)
    stream = torch.cuda.current_stream()
    P, sim, phi0, obs = make_sim(F, w, args.curv, args.storage, stream)
    flush = torch.empty(L2_FLUSH_BYTES // 4, dtype=torch.float32, device="cuda")

    sim.step(args.develop)
    for _ in range(args.warmup):  # by the call that is timed
        sim.step(1)
    torch.cuda.synchronize()
    st = sim.stats()
    n_fluid, n_if, N = int(st[0] + st[1]), int(st[1]), sim.N

    mass_start = sim.mass_total()
    # ---- timed region: K steps, each between events; L2 flushed before each
    if ws > 1:
        import torch.distributed as dist
        dist.barrier()
    torch.cuda.synchronize()
    clk = ClockSampler(local)
    time.sleep(0.15)
    t0 = time.time()
    ms = time_steps(sim, args.steps, stream, flush)
    t1 = time.time()
    ms, total_fluid = reduce_over_ranks(ms, n_fluid, "cuda")
    ms_per_step = ms / args.steps
    value = total_fluid * args.steps / (ms * 1e-3) / 1e6
    mass_end = sim.mass_total()
    drift = ((mass_end[0] + mass_end[1]) - (mass_start[0] + mass_start[1])) / (mass_start[0] + mass_start[1])

    # ---- per-phase device times (kernel by kernel, same state evolution)
    ph = phase_profile(sim, min(args.steps, 50), flush)
    clk.stop()
    clocks = clk.summary(t0, t1)

    # ---- curvature alone (LSQR) on the current state
    kap = torch.empty_like(sim.kappa)
    sim.curvature(F.CURV_LSQR, kap)
    cev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(20)]
    for a, b in cev:
        flush.fill_(1.0)
        a.record(stream)
        sim.curvature(F.CURV_LSQR, kap)
        b.record(stream)
    torch.cuda.synchronize()
    curv_ms = sum(a.elapsed_time(b) for a, b in cev) / len(cev)
    st2 = sim.stats()
    n_if_now, n_fp64 = int(st2[7]), int(st2[6])
    # ---- curvature alone (FD with K8 smoothing, Sec. II.A) on the same state
    try:
        sim.curvature(F.CURV_FD, kap)
        for a, b in cev:
            flush.fill_(1.0)
            a.record(stream)
            sim.curvature(F.CURV_FD, kap)
            b.record(stream)
        torch.cuda.synchronize()
        fd_ms = sum(a.elapsed_time(b) for a, b in cev) / len(cev)
        curv_fd = {"ms": fd_ms, "evals_per_s": n_if_now / (fd_ms * 1e-3), "includes": "normals + smoothing + FD"}
    except Exception as e:  # a side figure: the headline line is printed regardless
        curv_fd = {"error": str(e)[:200]}
    # ---- curvature alone (TR: triangle fan of PLIC points, Sec. II.B) on the same state
    try:
        sim.curvature(F.CURV_TR, kap)
        for a, b in cev:
            flush.fill_(1.0)
            a.record(stream)
            sim.curvature(F.CURV_TR, kap)
            b.record(stream)
        torch.cuda.synchronize()
        tr_ms = sum(a.elapsed_time(b) for a, b in cev) / len(cev)
        curv_tr = {"ms": tr_ms, "evals_per_s": n_if_now / (tr_ms * 1e-3), "includes": "normals + PLIC + fan"}
    except Exception as e:
        curv_tr = {"error": str(e)[:200]}

    # ---- mass reduction (FP64 partials) alone
    m0 = time.perf_counter()
    for _ in range(5):
        sim.mass_total()
    mass_ms = (time.perf_counter() - m0) * 1e3 / 5

    # ---- end to end through the public API with host buffers
    phi_host = phi0.cpu().pin_memory()
    obs_host = obs.cpu().pin_memory() if obs is not None else None
    sim.close()
    torch.cuda.synchronize()
    e0 = time.perf_counter()
    sim2 = F.Sim(P, phi0=phi_host.numpy(), obstacle=None if obs_host is None else obs_host.numpy(), stream=stream)
    sim2.step(args.steps)
    mtot, _ = sim2.mass_total()
    torch.cuda.synchronize()
    e_s = time.perf_counter() - e0
    h2d = N * 4 + (N if obs_host is not None else 0)
    e2e = {"value": n_fluid * args.steps / e_s / 1e6 * (ws if ws > 1 else 1), "unit": "MLUPS",
           "h2d_bytes_per_step": h2d / args.steps, "d2h_bytes_per_step": 16 / args.steps,
           "includes": "fsl_init from pinned host fill levels (upload, types, f = w_q), graph capture, K steps, "
                       "fsl_mass read back"}

    fused = args.curv == "lsqr"
    nb = algorithmic_bytes(n_fluid, n_if, n_fluid, fused=fused, pdf_bytes=4 if args.storage == "f32" else 2)
    roof = roofline_of(ph, nb, peaks, workload=args.workload if args.storage == "f32" else None, fused=fused)
    line = {"metric": METRIC, "value": value, "unit": "MLUPS", "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": ms_per_step, "higher_is_better": True, "scaling": "weak",
            "vs_baseline": None, "dtype": {"f32": "f32", "f16": "f16-offset/f32", "bf16": "bf16-offset/f32"}[args.storage],
            "data": "synthetic",
            "config": {"workload": args.workload, "grid": list(w["shape"][::-1]), "geometry": w["geometry"]["kind"],
                       "R": w["geometry"].get("R"), "sigma": w["sigma"], "tau": w["tau"], "curvature": args.curv,
                       "storage": args.storage, "l2": "flushed before every timed step (256 MiB write)",
                       "timed_from_step": args.develop + args.warmup,
                       "parallelism": f"replicas x{ws}" if ws > 1 else "single GPU"},
            "fluid_cells": n_fluid, "interface_cells": n_if, "mlups_domain": N * args.steps / (ms * 1e-3) / 1e6,
            "curvature_evals_per_s": n_if_now / (curv_ms * 1e-3), "curvature_ms": curv_ms,
            "curvature_fd": curv_fd, "curvature_tr": curv_tr,
            "lsqr_fp64_cells": n_fp64,
            "phases_ms": dict(zip(PHASES, [round(float(v), 5) for v in ph])),
            "mass_reduce_ms": mass_ms, "mass_drift_rel": drift, "roofline": roof, "e2e": e2e,
            "gpu_launches": kernels_per_step(args.curv, obs) * args.steps, "clocks": clocks}
    gs = None
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        gs = {"flags": sim2.flags_current().cpu().numpy(), "phi": sim2.phi.double().cpu().numpy()}
        sim2.curvature(F.CURV_LSQR)
        torch.cuda.synchronize()
        gs["kappa"] = sim2.kappa.double().cpu().numpy()
    sim2.close()
    del sim2, sim, phi0
    torch.cuda.empty_cache()
    if not args.no_side:
        side_steps = min(args.steps, 200)
        line["dense_pool"] = side_workload(F, S, "pool256", "f32", side_steps, stream, flush, peaks, S.SEED + rank)
        line["precision_forms"] = {
            st_: side_workload(F, S, "pool256", st_, side_steps, stream, flush, peaks, S.SEED + rank)
            for st_ in ("f16", "bf16")}
        lc = learned_curvature(F, S, stream, flush, peaks, S.SEED + rank, args.mlp_train, args.mlp_epochs,
                               min(args.steps, 100), batch=args.mlp_batch)
        held = lc.pop("heldout")
        net = lc.pop("net")
        line["learned_curvature"] = lc
        line["adjoint"] = adjoint_window(F, S, stream, S.SEED + rank)
        if not args.no_physics:
            t_ph = time.perf_counter()
            line["physics"] = physics_reports(F, S, stream, net)
            line["physics"]["seconds"] = time.perf_counter() - t_ph
        del net
    if gs is not None:
        line["cpu_baseline"] = oracle_sample(w, args.cpu_seconds, gpu_state=gs)
        line["cpu_all_cores"] = oracle_all_cores(w, min(args.cpu_seconds, 10.0))
        line["kappa_err_vs_fp64"] = line["cpu_baseline"].pop("kappa_check")
        if not args.no_side:
            line["learned_curvature"]["heldout_kappa_rel_err"] = heldout_errors(held)
            ref = adjoint_reference()
            adj = line["adjoint"]
            ref["rel_err_sigma"] = abs(adj["dL_dsigma"] - ref["dL_dsigma"]) / abs(ref["dL_dsigma"])
            ref["rel_err_theta"] = abs(adj["dL_dtheta"] - ref["dL_dtheta"]) / abs(ref["dL_dtheta"])
            adj["fp64_reference"] = ref
    if rank == 0:
        print(json.dumps(line), flush=True)
    if ws > 1:
        import torch.distributed as dist
        dist.barrier()
        dist.destroy_process_group()


def main():
    args = parse()
    if args.mlp_only:
        import torch
        from paper_1509_07691_gb300 import build, synthetic as S
        build.build()
        from paper_1509_07691_gb300 import fsl as F
        lc = learned_curvature(F, S, torch.cuda.current_stream(), None, {}, S.SEED, args.mlp_train, args.mlp_epochs, 0,
                               inference=False, batch=args.mlp_batch)
        held = lc.pop("heldout")
        lc.pop("net")
        lc["heldout_kappa_rel_err"] = heldout_errors(held)
        print(json.dumps({"learned_curvature": lc}))
        return
    if args.physics:
        import torch
        from paper_1509_07691_gb300 import build, synthetic as S
        build.build()
        from paper_1509_07691_gb300 import fsl as F
        print(json.dumps({"physics": physics_reports(F, S, torch.cuda.current_stream())}))
        return
    if args.adjoint_only:
        import torch
        from paper_1509_07691_gb300 import build, synthetic as S
        build.build()
        from paper_1509_07691_gb300 import fsl as F
        stream = torch.cuda.current_stream()
        print(json.dumps({"adjoint": adjoint_window(F, S, stream, S.SEED, reps=1, warm=0, checks=False)}))
        return
    if args.impl == "reference":
        run_reference(args)
    else:
        run_fsl(args)


if __name__ == "__main__":
    main()
