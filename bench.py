#!/usr/bin/env python
"""Benchmark of the constant-capacitance-model ground-state hot path on GB300.

Workload: the 16-dot 4x4-grid array, open, default algorithm (t = 1), a
100 x 100 raster over plungers 5 and 6 (seeded synthetic capacitances; the
paper benchmarks 16-dot 100 x 100 diagrams, Sec. VII).  One step = one whole
diagram through the C ABI: prep (continuous minimum + candidate set), the
candidate search, the FP64 recheck of flagged pixels, int8 charges + FP64
energies + flags written to HBM.

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference]

Prints one JSON line (rank 0).  Under torchrun every rank computes its own
diagrams (independent shards, no data-path collective; weak scaling).
"""
from __future__ import annotations

import argparse
import json
import math
import os
import statistics
import subprocess
import sys
import tempfile
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "CSD pixels/s (16-dot 100x100)"
UNIT = "pixels/s"
WORKLOAD = "grid16_4x4_open_t1_100x100"
PAPER_CONTEXT = ("paper: 16-dot 100x100 diagram in < 1 s (> 1e4 px/s) with the JAX "
                 "default core on a GTX 1080 Ti (Sec. VII) -- other hardware, context only")


# --------------------------------------------------------------------------
# clocks during the timed region
# --------------------------------------------------------------------------
class ClockSampler:
    FIELDS = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu_index=0, period_ms=100):
        self.path = tempfile.mktemp(prefix="qa_clocks_", suffix=".csv")
        self.proc = None
        self.gpu = gpu_index
        self.period = period_ms

    def start(self):
        try:
            self.fh = open(self.path, "w")
            self.proc = subprocess.Popen(
                ["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.FIELDS}",
                 "--format=csv,noheader,nounits", "-lms", str(self.period)],
                stdout=self.fh, stderr=subprocess.DEVNULL)
        except Exception:
            self.proc = None
        return self

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"],
                    "samples": 0}
        self.proc.terminate()
        try:
            self.proc.wait(timeout=5)
        except Exception:
            self.proc.kill()
        self.fh.close()
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
                if v.lower().startswith("active"):
                    reasons.add(nm)
        os.unlink(self.path)
        return {"sm_mhz": statistics.median(sm) if sm else None,
                "sm_max_mhz": max(smax) if smax else None,
                "reasons": sorted(reasons), "samples": len(sm)}


# --------------------------------------------------------------------------
def search_traffic():
    """dram read+write bytes per launch of the ground-state kernel (prep +
    search) from the committed ncu summary, or None when the kernel sources
    changed since that capture."""
    import hashlib
    import re
    prof = os.path.join(ROOT, "profiles", "ground_state_kernel_grid16_100x100.md")
    if not os.path.exists(prof):
        return None
    text = open(prof).read()
    m_hash = re.search(r"kernel_source_sha256_16: ([0-9a-f]{16})", text)
    m_traf = re.search(r"\| traffic_bytes_per_launch \| (\d+) \|", text)
    if not (m_hash and m_traf):
        return None
    csrc = os.path.join(ROOT, "paper_2404_04994_gb300", "csrc")
    h = hashlib.sha256()
    for f in ("qa_search.cuh", "qa_sphere.cuh", "qa_gs_tiles.cuh", "qa_pixels.cu",
              "qa_kernels_gs.cu", "qa_device.cuh", "qa_prep.cuh"):
        h.update(open(os.path.join(csrc, f), "rb").read())
    return int(m_traf.group(1)) if h.hexdigest()[:16] == m_hash.group(1) else None


def workload(rank=0):
    from paper_2404_04994_gb300 import inputs
    cfg = inputs.grid16(W=100, H=100, t=1.0)
    return cfg


def oracle_rate(cfg, budget_s, rows=None, threads=None):
    """FP64 oracle pixels/s on all host cores (or `threads`) over a bounded
    sample of rows."""
    import oracle
    W = cfg["raster"]["W"]
    cores = threads or os.cpu_count() or 1
    # calibrate on one block of pixels, then size the sample to the budget
    t0 = time.perf_counter()
    oracle.ground_state(cfg["Cdd"], cfg["Cgd"], raster=cfg["raster"], t=cfg["t"],
                        pixels=(0, cores), n_threads=cores)
    per_px = (time.perf_counter() - t0) / cores
    if rows is None:
        npx = max(cores, min(W * cfg["raster"]["H"], int(budget_s / max(per_px, 1e-9))))
    else:
        npx = rows * W
    p0 = (cfg["raster"]["H"] // 2) * W
    p1 = min(p0 + npx, W * cfg["raster"]["H"])
    t0 = time.perf_counter()
    oracle.ground_state(cfg["Cdd"], cfg["Cgd"], raster=cfg["raster"], t=cfg["t"],
                        pixels=(p0, p1), n_threads=cores)
    dt = time.perf_counter() - t0
    return (p1 - p0) / dt, cores, p1 - p0, dt


def run_reference(args):
    from paper_2404_04994_gb300 import dist
    rank, local, world = dist.env_rank()
    if rank != 0:
        return
    cfg = workload()
    cores = os.cpu_count() or 1
    budget = 120.0 / max(1, args.steps + args.warmup)   # whole run ~2 minutes
    for _ in range(args.warmup):
        oracle_rate(cfg, budget)
    rates, total_px, total_t = [], 0, 0.0
    for _ in range(args.steps):
        r, cores, npx, dt = oracle_rate(cfg, budget)
        rates.append(r)
        total_px += npx
        total_t += dt
    value = total_px / total_t
    line = {"impl": "reference", "metric": METRIC, "value": value, "unit": UNIT,
            "n_gpus": args.gpus, "steps": args.steps, "warmup": args.warmup,
            "ms_per_step": 1e3 * total_t / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
            "config": {"workload": WORKLOAD, "n_dot": 16, "pixels": 10000,
                       "threshold": 1.0, "sample": "contiguous pixel rows from the "
                       "middle of the raster, sized per step to the time budget"},
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": cores,
                             "kind": "oracle",
                             "sample": f"{total_px} pixels over {args.steps} steps"},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0,
                    "d2h_bytes_per_step": 0}}
    print(json.dumps(line))


# --------------------------------------------------------------------------
def run_ours(args):
    import numpy as np
    import torch

    from paper_2404_04994_gb300 import api, dist

    rank, local, world = dist.init()
    torch.cuda.set_device(local)
    peaks = {}
    pk = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(pk):
        peaks = json.load(open(pk))
    cfg = workload(rank)
    P = cfg["raster"]["W"] * cfg["raster"]["H"]
    n_dot = cfg["Cdd"].shape[0]
    m = api.Model(cfg["Cdd"], cfg["Cgd"])
    h = m.handle
    ras = cfg["raster"]
    dev = torch.device("cuda", local)
    out_n = torch.empty((P, n_dot), dtype=torch.int8, device=dev)
    out_U = torch.empty(P, dtype=torch.float64, device=dev)
    out_f = torch.empty(P, dtype=torch.uint8, device=dev)
    flush = torch.empty(256 * 1024 * 1024 // 4, dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream()

    def step():
        api.qa_ground_state_open(h, ras, 1.0, out_n, out_U, out_f, stream)

    for _ in range(max(3, args.warmup)):
        step()
    torch.cuda.synchronize()
    st0 = m.stats()

    # ---- timed region: K diagrams, L2 flushed between them ----
    starts = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    ends = [torch.cuda.Event(enable_timing=True) for _ in range(args.steps)]
    clocks = ClockSampler(gpu_index=local).start()
    time.sleep(0.25)
    dist.barrier()
    torch.cuda.synchronize()
    for i in range(args.steps):
        flush.zero_()
        starts[i].record(stream)
        step()
        ends[i].record(stream)
    torch.cuda.synchronize()
    dist.barrier()
    clk = clocks.stop()
    dev_ms = sum(s.elapsed_time(e) for s, e in zip(starts, ends))
    dev_ms = dist.max_over_ranks(dev_ms)
    ms_per_step = dev_ms / args.steps
    value = world * P / (ms_per_step * 1e-3)

    # ---- roofline: the search kernel timed alone by the library's events ----
    api.qa_model_set_timing(h, True)
    search_ms, prep_ms, recheck_ms = [], [], []
    for _ in range(20):
        flush.zero_()
        step()
        s = m.stats()
        search_ms.append(s["ms_search"])
        prep_ms.append(s["ms_prep"])
        recheck_ms.append(s["ms_recheck"])
    api.qa_model_set_timing(h, False)
    st = m.stats()
    L1, L2 = st["inner_bits"], st["middle_bits"]
    # FP32 lane-operations of the sphere search per evaluated child: a node's
    # four children take two rows of four table sums and the centre (10), the
    # three further row sums (3), six squares with their additions (12) and
    # three gradient terms
    ops_per_child = 28.0 / 4.0
    ops = st["evaluated"] * ops_per_child
    ms_s = statistics.mean(a + b for a, b in zip(prep_ms, search_ms))
    achieved = ops / (ms_s * 1e-3) / 1e12
    sm_max = (clk.get("sm_max_mhz") or peaks.get("sm_max_mhz") or 2070.0)
    n_sm = torch.cuda.get_device_properties(dev).multi_processor_count
    peak = n_sm * 128 * sm_max * 1e6 / 1e12   # FP32 lanes x clock
    # the same diagram searched exhaustively (every one of the 2^16 candidates
    # at the split walk's 3.375 lane-operations): what the search saves
    exh = st["candidates"] * 3.375 / (ms_s * 1e-3) / 1e12
    roofline = {"bound": "alu", "achieved": round(achieved, 3), "peak": round(peak, 3),
                "unit": "Tops/s", "frac": round(achieved / peak, 4), "traffic": search_traffic(),
                "kernel": "k_pixels<16,open,sphere> (prep, sphere search and outputs)",
                "ops_per_launch": ops, "ops_per_evaluated_child": ops_per_child,
                "exhaustive_equivalent_tops": round(exh, 3),
                # one kernel prepares and searches
                "kernel_ms": round(ms_s, 5),
                "resolve_recheck_ms": round(statistics.mean(recheck_ms), 5),
                "peak_basis": f"{n_sm} SMs x 128 FP32 lanes x {sm_max:.0f} MHz (of nominal "
                              "unit counts and max clock; MEASURED_PEAKS.json has no FP32 figure)"}

    # ---- end to end: host matrices in, host charge map out ----
    # Every step uploads the model from host memory (the library stages it
    # in pinned memory and copies it in stream order), runs the call and
    # reads the charge map, energies and flags back into pinned host memory;
    # the three outputs sit in one device block, so one copy brings them
    # back.  Each step is timed with CUDA events from before the upload to
    # after the read-back has landed, with the L2 flushed between steps
    # (outside the events) as for the device-resident number; the host
    # prepares step k + 1 while the flush runs.
    Cdd, Cgd = cfg["Cdd"], cfg["Cgd"]
    ras_c = api.make_raster(ras, Cgd.shape[1])
    nb_n, nb_U = P * n_dot, P * 8
    off_U = (nb_n + 7) // 8 * 8
    nbytes = off_U + nb_U + P
    dblk = torch.empty(nbytes, dtype=torch.uint8, device=dev)
    hblk = torch.empty(nbytes, dtype=torch.uint8, pin_memory=True)
    d_n = dblk[:nb_n].view(torch.int8).view(P, n_dot)
    d_U = dblk[off_U:off_U + nb_U].view(torch.float64)
    d_f = dblk[off_U + nb_U:]
    ke = max(3, min(args.steps, 200))
    e0 = [torch.cuda.Event(enable_timing=True) for _ in range(ke)]
    e1 = [torch.cuda.Event(enable_timing=True) for _ in range(ke)]
    torch.cuda.synchronize()
    for i in range(ke):
        flush.zero_()
        e0[i].record(stream)
        api.qa_model_update_async(h, Cdd, Cgd, stream)
        api.qa_ground_state_open(h, ras_c, 1.0, d_n, d_U, d_f, stream)
        hblk.copy_(dblk, non_blocking=True)
        e1[i].record(stream)
    torch.cuda.synchronize()
    e2e_s = dist.max_over_ranks(sum(x.elapsed_time(y) for x, y in zip(e0, e1)) * 1e-3 / ke)
    bi = Cdd.nbytes + Cgd.nbytes + 3 * 8 * Cgd.shape[1] + 4 * 8 + 2 * 4
    bo = nb_n + nb_U + P

    extra = {"paper_context": PAPER_CONTEXT,
             "flagged_per_diagram": st["flagged"], "near_tie": st["near_tie"],
             "boundary": st["boundary"], "qp_pixels": st["qp_pixels"],
             "unresolved": st["unresolved"], "team": st["team"],
             "split": [L1, L2], "candidates_per_diagram": st["candidates"],
             "evaluated_slots_per_diagram": st["evaluated"],
             "gray_equivalent_gflop_per_diagram": st["candidates"] * (2 * 16 + 4) / 1e9}
    if not args.no_extra and world == 1:
        extra.update(extra_measurements(api, torch, flush, args))

    cpu = None
    if rank == 0 and world == 1:
        r, cores, npx, dt = oracle_rate(cfg, budget_s=20.0)
        r1, _, npx1, dt1 = oracle_rate(cfg, budget_s=6.0, threads=1)
        cpu = {"value": r, "unit": UNIT, "cores": cores, "kind": "oracle",
               "sample": f"{npx} contiguous pixels of the same diagram, FP64 oracle on "
                         f"{cores} host threads, {dt:.1f} s wall",
               "single_core": {"value": r1, "unit": UNIT, "cores": 1,
                               "sample": f"{npx1} contiguous pixels, one host thread, "
                                         f"{dt1:.1f} s wall"}}

    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world,
            "steps": args.steps, "warmup": args.warmup, "ms_per_step": ms_per_step,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None,
            "dtype": "f32", "data": "synthetic",
            "config": {"workload": WORKLOAD, "n_dot": 16, "pixels": P, "threshold": 1.0,
                       "parallelism": f"replicas x{world}",
                       "l2": "256 MiB buffer written between steps (outside the "
                             "per-step events)"},
            "roofline": roofline, "cpu_baseline": cpu,
            "e2e": {"value": world * P / e2e_s, "unit": UNIT,
                    "h2d_bytes_per_step": int(bi), "d2h_bytes_per_step": int(bo)},
            # per step: k_pixels (prep, search and outputs) and k_lists (close
            # candidates, near-tie resolve and FP64 recheck)
            "gpu_launches": 2 * args.steps, "clocks": clk, "extra": extra}
    if rank == 0:
        print(json.dumps(line))
    m.close()
    dist.finalize()


def extra_measurements(api, torch, flush, args):
    """Secondary numbers (not the headline): thresholded search, smaller
    arrays, the soft occupation and one gradient step."""
    import numpy as np

    from paper_2404_04994_gb300 import inputs
    out = {}

    def timed(fn, reps=30):
        for _ in range(3):
            fn()
        ev = []
        for _ in range(reps):
            flush.zero_()
            # keep the device busy (about 0.2 ms) while the host marshals the
            # call, so the events time the device work and not the binding
            torch.cuda._sleep(400000)
            a = torch.cuda.Event(enable_timing=True)
            b = torch.cuda.Event(enable_timing=True)
            a.record()
            fn()
            b.record()
            ev.append((a, b))
        torch.cuda.synchronize()
        return statistics.mean(a.elapsed_time(b) for a, b in ev)

    cfg = inputs.grid16(t=0.5)
    m = api.Model(cfg["Cdd"], cfg["Cgd"])
    ms = timed(lambda: m.ground_state_open(cfg["raster"], threshold=0.5))
    out["grid16_t0.5_pixels_per_s"] = 1e4 / (ms * 1e-3)
    out.update(search_profile(api, m, lambda: m.ground_state_open(cfg["raster"], threshold=0.5),
                              flush, "grid16_t0.5"))
    # closed 16-dot diagram, N_hat = 16 (every pixel needs the QP)
    ms = timed(lambda: m.ground_state_closed(cfg["raster"], 16, threshold=1.0))
    out["grid16_closed_pixels_per_s"] = 1e4 / (ms * 1e-3)
    out["grid16_closed_ms"] = ms
    st = m.stats()
    out["grid16_closed_qp_pixels"] = st["qp_pixels"]
    out["grid16_closed_fp64_rechecks"] = st["boundary"]
    # the paper's benchmark shape (Sec. VII): 16 dots, 10^4 random gate-voltage
    # vectors (no raster coherence), open and closed N_hat = 16
    Vd = torch.tensor(inputs.random_points(16, 10000, seed=11), device="cuda")
    for closed in (False, True):
        tag = "points16_closed" if closed else "points16_open"
        fn = ((lambda: m.ground_state_points(Vd, closed=True, n_charges=16)) if closed
              else (lambda: m.ground_state_points(Vd)))
        ms = timed(fn)
        st = m.stats()
        out[f"{tag}_pixels_per_s"] = 1e4 / (ms * 1e-3)
        out[f"{tag}_qp_pixels"] = st["qp_pixels"]
        out[f"{tag}_flagged"] = st["flagged"]
    m.close()
    for name, c, closed in (("double_dot_100x100", inputs.double_dot(), False),
                            ("chain4_open_200x200", inputs.chain4(), False),
                            ("chain4_closed_200x200", inputs.chain4(closed=True), True)):
        m = api.Model(c["Cdd"], c["Cgd"])
        P = c["raster"]["W"] * c["raster"]["H"]
        if closed:
            ms = timed(lambda: m.ground_state_closed(c["raster"], 4))
        else:
            ms = timed(lambda: m.ground_state_open(c["raster"]))
        out[f"{name}_pixels_per_s"] = P / (ms * 1e-3)
        # the brute-force row of Table I on the same raster, for comparison
        r = c["raster"]
        corners = [np.asarray(r["V0"]) + x * np.asarray(r["u"]) + y * np.asarray(r["w"])
                   for x in (r["x0"], r["x1"]) for y in (r["y0"], r["y1"])]
        cmax = max(float(np.max(np.asarray(c["Cgd"]) @ v)) for v in corners)
        nmax = int(math.ceil(max(cmax, 0.0))) + 2
        if closed:
            ms_b = timed(lambda: m.brute_force_closed(r, 4), reps=5)
        else:
            ms_b = timed(lambda: m.brute_force_open(r, nmax), reps=5)
        out[f"{name}_brute_force_pixels_per_s"] = P / (ms_b * 1e-3)
        if not closed:
            out[f"{name}_brute_force_n_max"] = nmax
        m.close()
    out.update(batch_measurements(api, torch, flush))
    try:
        from paper_2404_04994_gb300 import autograd as qag
        for kT in (0.01, 0.05):
            c = inputs.grid8(kT=kT)
            # the fused library step (graph replay and plain launches), and
            # the same step through torch autograd + torch.optim.Adam
            ms_step = qag.time_grad_step(c, kT, flush=flush)
            out[f"grad_step_ms_grid8_kT{kT:g}"] = ms_step
            out[f"grad_step_plain_ms_grid8_kT{kT:g}"] = qag.time_grad_step(c, kT, flush=flush,
                                                                         graph=False)
            out[f"grad_step_autograd_ms_grid8_kT{kT:g}"] = qag.time_grad_step(
                c, kT, flush=flush, fused=False)
    except ImportError:
        pass
    return out


def search_profile(api, m, fn, flush, tag):
    """Device-counted candidates and evaluated slots of one call, with the
    library's per-kernel times (prep, search, resolve + recheck) and the
    search's lane-ops rate on the same basis as the headline roofline."""
    api.qa_model_set_timing(m.handle, True)
    ks, kp, kr = [], [], []
    for _ in range(20):
        flush.zero_()
        fn()
        s = m.stats()
        ks.append(s["ms_search"])
        kp.append(s["ms_prep"])
        kr.append(s["ms_recheck"])
    api.qa_model_set_timing(m.handle, False)
    st = m.stats()
    L1, L2 = st["inner_bits"], st["middle_bits"]
    # (no inner slots: the sphere search, 7 operations a child as above)
    ops = st["evaluated"] * (3.0 + (L1 + L2 + 3.0) / (1 << L1) if L1 else 7.0)
    ms = statistics.mean(ks)
    return {f"{tag}_candidates": st["candidates"], f"{tag}_evaluated_slots": st["evaluated"],
            f"{tag}_search_ms": ms, f"{tag}_prep_ms": statistics.mean(kp),
            f"{tag}_resolve_recheck_ms": statistics.mean(kr),
            f"{tag}_candidates_per_s": st["candidates"] / (ms * 1e-3),
            f"{tag}_search_tops": ops / (ms * 1e-3) / 1e12, f"{tag}_team": st["team"]}


def batch_measurements(api, torch, flush):
    """The 4096-array batch (N ~ U{2..16}, 64^2 / 128^2 rasters, open or
    closed with N_hat = N): one graph-captured batched run versus the plain
    form (one single-array call per array), pixels/s of each."""
    from paper_2404_04994_gb300 import inputs
    specs = inputs.batch(4096)
    b = api.Batch(specs)
    b.run()
    torch.cuda.synchronize()
    st = b.stats()
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        b.run(s)
    torch.cuda.current_stream().wait_stream(s)
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        b.run()
    times = []
    for _ in range(3):
        flush.zero_()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record()
        g.replay()
        e1.record()
        torch.cuda.synchronize()
        times.append(e0.elapsed_time(e1))
    ms_batch = min(times)
    # plain form: one call per array, outputs preallocated, after a warm-up pass
    def plain():
        for sp, m, (n, U, f) in zip(specs, b.models, b.outputs):
            if sp["closed"]:
                api.qa_ground_state_closed(m.handle, sp["raster"], sp["t"], sp["n_charges"],
                                           n, U, f)
            else:
                api.qa_ground_state_open(m.handle, sp["raster"], sp["t"], n, U, f)
    plain()
    torch.cuda.synchronize()
    flush.zero_()
    e0 = torch.cuda.Event(enable_timing=True)
    e1 = torch.cuda.Event(enable_timing=True)
    e0.record()
    plain()
    e1.record()
    torch.cuda.synchronize()
    ms_plain = e0.elapsed_time(e1)
    out = {"batch4096_pixels": b.pixels, "batch4096_ms": ms_batch,
           "batch4096_pixels_per_s": b.pixels / (ms_batch * 1e-3),
           "batch4096_plain_ms": ms_plain,
           "batch4096_plain_pixels_per_s": b.pixels / (ms_plain * 1e-3),
           "batch4096_candidates": st["candidates"], "batch4096_flagged": st["flagged"],
           "batch4096_unresolved": st["unresolved"]}
    del g
    b.close()
    # autotuned: threshold and team per (N, form) from 24 x 24 samples
    from paper_2404_04994_gb300 import autotune
    import time
    t0 = time.perf_counter()
    table = autotune.tune(specs, sample_side=24, arrays_per_group=4)
    tune_s = time.perf_counter() - t0
    tb = api.Batch(autotune.apply(specs, table))
    tb.run()
    torch.cuda.synchronize()
    gt = torch.cuda.CUDAGraph()
    s2 = torch.cuda.Stream()
    s2.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s2):
        tb.run(s2)
    torch.cuda.current_stream().wait_stream(s2)
    with torch.cuda.graph(gt):
        tb.run()
    tt = []
    for _ in range(3):
        flush.zero_()
        e0 = torch.cuda.Event(enable_timing=True)
        e1 = torch.cuda.Event(enable_timing=True)
        e0.record()
        gt.replay()
        e1.record()
        torch.cuda.synchronize()
        tt.append(e0.elapsed_time(e1))
    tst = tb.stats()
    out.update({"batch4096_tuned_ms": min(tt),
                "batch4096_tuned_pixels_per_s": tb.pixels / (min(tt) * 1e-3),
                "batch4096_tuned_candidates": tst["candidates"],
                "batch4096_tuned_unresolved": tst["unresolved"],
                "autotune_s": tune_s,
                "autotune_table": {f"{'closed' if c else 'open'}{n}": [e["threshold"], e["team"]]
                                   for (n, c), e in sorted(table.items())}})
    del gt
    tb.close()
    return out


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=500)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", choices=["ours", "reference"], default="ours")
    ap.add_argument("--no-extra", action="store_true")
    args = ap.parse_args()
    if args.impl == "reference":
        run_reference(args)
    else:
        run_ours(args)


if __name__ == "__main__":
    main()
