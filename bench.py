#!/usr/bin/env python
"""Throughput of the FFT-based diffuse-scattering calculation on one GB300 (or N replicas).

Workload (the compositional + magnetic configuration): cubic cell a = 10 A with the 16
pyrochlore sites, 20x20x20 supercell, Bernoulli(0.3) occupancies and unit spins from
vMF(kappa = 2) about seeded per-site axes, <j0> magnetic form factor (A=0.4 a=15 B=0.6 b=5 C=0
c=1 D=0), Q grid |h|,|k|,|l| <= 6 in steps of 1/20 (241^3 = 13,997,521 voxels).  One step =
the whole hot path for both volumes: per-site FFTs + recombination + |F|^2 (nuclear, diffuse
mode) and per-site/per-component FFTs + recombination + perpendicular projection (magnetic,
total mode), FP32 arithmetic; the two independent volumes run on two streams (--streams 1:
one after the other).  Metric: intensity voxels/s (both volumes counted), checked against the
FP64 path of the same kernels (<= 1e-5 of peak).

  python bench.py [--gpus N] [--steps K] [--warmup W] [--impl ours|reference] [--streams 1|2]
Under torchrun each rank runs an independent replica on its own GPU (the workload does not
shard); rank 0 prints one JSON line.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import subprocess
import sys
import threading
import time

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "intensity voxels/s at <=1e-5 rel err vs plain FP64 GPU path"
UNIT = "voxels/s"
HMAX, NCELL, NSITE = 6.0, 20, 16
FP32_FMA_LANES_PER_SM, NUM_SMS = 128, 152
# dram__bytes_read.sum + dram__bytes_write.sum of one launch of the magnetic recombination on
# this workload, from an ncu capture of the current kernel (profiles/); None when the kernel has
# changed since the capture
MAG_KERNEL = "k_recomb_rows<float,3,2,true,false>"
# dram__bytes_read.sum + dram__bytes_write.sum of one launch of the kernel above (ncu,
# profiles/k_recomb_rows_pyrochlore_20cubed.md): the reads are the spectra read once; the volume
# written is still in L2 when the kernel ends (written back later, during the next step's flush)
MAG_KERNEL_TRAFFIC = 1778688 + 221440
MAG_KERNEL_TRAFFIC_SOURCE = ("ncu capture of k_recomb_rows<float,3,2,true,false> on this workload: 1.78 MB read "
                             "(the spectra, once) + 0.22 MB written to DRAM before the kernel ended; the rest of the "
                             "56 MB volume was still in L2")


def workload_config(extra=None):
    c = {"workload": "pyrochlore occupancy+magnetic, 16 sites, 20x20x20 cells, |hkl|<=6 step 1/20 "
                     "(241^3 voxels), nuclear diffuse + magnetic total volumes",
         "cells": [NCELL] * 3, "nsite": NSITE, "voxels_per_volume": 241 ** 3, "volumes_per_step": 2,
         "l2": "256 MB memset between steps, outside the per-step events"}
    if extra:
        c.update(extra)
    return c


def dist_env():
    ws = int(os.environ.get("WORLD_SIZE", "1"))
    rank = int(os.environ.get("RANK", "0"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return ws, rank, local


def init_dist(backend):
    ws, rank, local = dist_env()
    if ws > 1:
        import torch.distributed as dist
        dist.init_process_group(backend=backend)
    return ws, rank, local


def max_over_ranks(x, device=None):
    ws, _, _ = dist_env()
    if ws == 1:
        return x
    import torch
    import torch.distributed as dist
    t = torch.tensor([float(x)], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def barrier(device=None):
    ws, _, _ = dist_env()
    if ws > 1:
        import torch.distributed as dist
        if device is not None:
            dist.barrier(device_ids=[device.index])
        else:
            dist.barrier()


class ClockSampler:
    """nvidia-smi clocks / throttle reasons sampled every 20 ms while running."""
    FIELDS = ("clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,"
              "clocks_event_reasons.hw_slowdown,clocks_event_reasons.hw_thermal_slowdown,"
              "clocks_event_reasons.sw_thermal_slowdown,clocks_event_reasons.sw_power_cap")

    def __init__(self, index):
        self.index = index
        self.rows = []
        self.proc = None

    def start(self):
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.index), "--query-gpu=" + self.FIELDS,
                                          "--format=csv,noheader,nounits", "-lms", "20"],
                                         stdout=subprocess.PIPE, stderr=subprocess.DEVNULL, text=True)
            self.t = threading.Thread(target=self._read, daemon=True)
            self.t.start()
        except OSError:
            self.proc = None

    def _read(self):
        for line in self.proc.stdout:
            parts = [p.strip() for p in line.split(",")]
            if len(parts) >= 8:
                self.rows.append(parts)

    def stop(self):
        if self.proc:
            self.proc.terminate()
            try:
                self.proc.wait(timeout=5)
            except subprocess.TimeoutExpired:
                self.proc.kill()
        out = {"sm_mhz": None, "sm_max_mhz": None, "reasons": [], "samples": len(self.rows)}
        if not self.rows:
            return out
        try:
            sm = [float(r[0]) for r in self.rows]
            out["sm_mhz"] = statistics.median(sm)
            out["sm_max_mhz"] = max(float(r[1]) for r in self.rows)
            out["power_w_max"] = max(float(r[2]) for r in self.rows)
        except ValueError:
            pass
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        reasons = set()
        for r in self.rows:
            for n, v in zip(names, r[4:8]):
                if v.strip().lower() == "active":
                    reasons.add(n)
        out["reasons"] = sorted(reasons)
        return out


def measured_peaks():
    try:
        with open(os.path.join(ROOT, "MEASURED_PEAKS.json")) as f:
            return json.load(f), "measured"
    except OSError:
        return {"hbm_gbs": 6800.0, "bf16_tflops": 1900.0, "sm_max_mhz": 2070.0}, "fallback"


# ----------------------------------------------------------------------------------------------
# the CPU oracle, timed on the host cores (cpu_baseline leg and --impl reference)
# ----------------------------------------------------------------------------------------------

def host_cpu():
    """(cores, model) of the host: os.cpu_count() and the model name from lscpu or /proc/cpuinfo."""
    model = None
    try:
        out = subprocess.run(["lscpu"], capture_output=True, text=True, timeout=10).stdout
        for line in out.splitlines():
            if line.lower().startswith("model name"):
                model = line.split(":", 1)[1].strip()
                break
    except (OSError, subprocess.SubprocessError):
        pass
    if model is None:
        try:
            with open("/proc/cpuinfo") as f:
                for line in f:
                    if line.lower().startswith(("model name", "cpu part")):
                        model = line.split(":", 1)[1].strip()
                        break
        except OSError:
            pass
    return os.cpu_count() or 1, model


def _pool_init():
    sys.path.insert(0, ROOT)
    import synthetic  # noqa: F401
    from oracle import core  # noqa: F401


def _pool_zones(zones):
    """One worker's share: the oracle's FFT method (numpy FP64) for both volumes on `zones`."""
    import synthetic as syn
    m = syn.pyrochlore_occ_mag()
    return oracle_sample_step(m, syn.magnetic_view(m), zones)


def oracle_pool(nproc):
    """A pool of nproc processes started with spawn (safe after CUDA has been initialised)."""
    import multiprocessing as mp
    pool = mp.get_context("spawn").Pool(nproc, initializer=_pool_init)
    pool.map(_pool_zones, [zone_voxels(1)[:1]] * nproc)   # import and first-touch outside the timing
    return pool


def pool_zone_rate(pool, nproc, nzones):
    """Voxels per second of the oracle's FFT method over nzones whole H zones spread on the pool."""
    zones = zone_voxels(nzones)
    parts = [zones[i::nproc] for i in range(nproc) if zones[i::nproc]]
    t0 = time.perf_counter()
    vox = sum(pool.map(_pool_zones, parts))
    dt = time.perf_counter() - t0
    return vox, dt

def oracle_sample_step(m, mm, zones):
    """The oracle's FFT method (numpy, FP64) for both volumes on the voxels of `zones`."""
    import numpy as np
    from oracle import core
    G = np.concatenate([z for z in zones])
    core.occupancy_intensity_fft(m, G, core.DIFFUSE)
    core.magnetic_intensity_fft(mm, G, core.TOTAL)
    return 2 * G.shape[0]


def zone_voxels(count):
    import numpy as np
    rng = np.random.default_rng(12345)
    out = []
    k = np.stack(np.meshgrid(*(np.arange(NCELL),) * 3, indexing="ij"), -1).reshape(-1, 3)
    for _ in range(count):
        H = rng.integers(-6, 6, 3)
        out.append(H[None, :] * NCELL + k)
    return out


def cpu_baseline(seconds=12.0):
    """The oracle's FFT method on whole H zones of the workload, spread over a process pool with one
    process per host core (each numpy FFT single-threaded)."""
    nproc, model = host_cpu()
    pool = oracle_pool(nproc)
    try:
        vox, dt = pool_zone_rate(pool, nproc, nproc)
        nz = max(nproc, int(nproc * seconds / max(dt, 1e-3)))
        vox, dt = pool_zone_rate(pool, nproc, nz)
    finally:
        pool.close()
        pool.join()
    return {"value": vox / dt, "unit": UNIT, "cores": nproc, "cpu_model": model, "kind": "oracle",
            "sample": "%d whole H zones (%d voxels per volume, both volumes) of the workload by the oracle's "
                      "FFT method (numpy FP64), %d processes, %.1f s" % (nz, vox // 2, nproc, dt)}


def cpu_direct_rate(m, hkl, mode, disorder="disp"):
    """Voxels per second of the oracle's direct sum (C, OpenMP over Q on every host core)."""
    from oracle import core
    t0 = time.perf_counter()
    if disorder == "disp":
        core.displacive_intensity_direct(m, hkl, mode)
    dt = time.perf_counter() - t0
    return hkl.shape[0] / dt, dt, core.oracle_threads()


def run_reference(args):
    ws, rank, local = init_dist("gloo")
    if rank != 0:
        return 0
    nproc, model = host_cpu()
    pool = oracle_pool(nproc)
    try:
        # size one step to ~1.5 s of CPU work on the pool
        vox, dt = pool_zone_rate(pool, nproc, nproc)
        nz = max(nproc, int(nproc * 1.5 / max(dt, 1e-3)))
        for _ in range(args.warmup):
            pool_zone_rate(pool, nproc, nz)
        el, vox = 0.0, 0
        for _ in range(args.steps):
            v, dt = pool_zone_rate(pool, nproc, nz)
            vox += v
            el += dt
    finally:
        pool.close()
        pool.join()
    value = vox / el
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1e3 * el / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic", "impl": "reference",
            "config": workload_config({"reference": "CPU FP64 oracle (FFT method, numpy), bounded sample of %d "
                                                    "H zones per step on %d processes" % (nz, nproc)}),
            "cpu_baseline": {"value": value, "unit": UNIT, "cores": nproc, "cpu_model": model, "kind": "oracle",
                             "sample": "%d whole H zones per step, both volumes, %d processes" % (nz, nproc)},
            "e2e": {"value": value, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line))
    return 0


# ----------------------------------------------------------------------------------------------
# the GPU path
# ----------------------------------------------------------------------------------------------

def run_ours(args):
    import numpy as np
    import torch

    ws, rank, local = init_dist("nccl")
    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    import paper_1809_07088_gb300 as ds
    import synthetic as syn

    m = syn.pyrochlore_occ_mag()
    mm = syn.magnetic_view(m)
    q = (m.qgrid.h0, m.qgrid.step, m.qgrid.count)
    nvox = m.qgrid.nvox
    ctx = ds.Context(local)
    lm_n = ds.Model(ctx, m.lattice, m.sites, m.cells, 1, m.scat_len, m.ff_kind, m.ff_coef)
    lm_m = ds.Model(ctx, mm.lattice, mm.sites, mm.cells, 1, mm.scat_len, mm.ff_kind, mm.ff_coef)
    occ_h = torch.from_numpy(np.ascontiguousarray(m.occ)).pin_memory()
    spin_h = torch.from_numpy(np.ascontiguousarray(m.spins)).pin_memory()
    occ_d, spin_d = occ_h.to(dev), spin_h.to(dev)
    lm_n.upload_occupancy(occ_d)
    lm_m.upload_spins(spin_d)
    I_n = torch.empty(m.qgrid.count, dtype=torch.float32, device=dev)
    I_m = torch.empty(m.qgrid.count, dtype=torch.float32, device=dev)
    stream = torch.cuda.current_stream(dev)

    side = [torch.cuda.Stream(dev), torch.cuda.Stream(dev)] if args.streams == 2 else None
    fork, join = torch.cuda.Event(), [torch.cuda.Event(), torch.cuda.Event()]

    def step(prec=ds.DS_FP32, outs=(I_n, I_m), single=False):
        if side is None or single:
            lm_n.intensity(q, out=outs[0], disorder=ds.DS_OCC, mode=ds.DS_DIFFUSE, precision=prec)
            lm_m.intensity(q, out=outs[1], disorder=ds.DS_SPIN, mode=ds.DS_TOTAL, precision=prec)
            return
        # the two independent volumes on two streams, forked from and joined back to the current one
        cur = torch.cuda.current_stream(dev)
        fork.record(cur)
        for s_, j_, (lm_, o_, dis, mode) in zip(side, join, ((lm_n, outs[0], ds.DS_OCC, ds.DS_DIFFUSE),
                                                            (lm_m, outs[1], ds.DS_SPIN, ds.DS_TOTAL))):
            s_.wait_event(fork)
            with torch.cuda.stream(s_):
                lm_.intensity(q, out=o_, disorder=dis, mode=mode, precision=prec)
            j_.record(s_)
            cur.wait_event(j_)

    flush = torch.empty(256 << 20, dtype=torch.uint8, device=dev)
    clocks = ClockSampler(local)
    clocks.start()
    for _ in range(args.warmup):
        step()
    torch.cuda.synchronize(dev)

    buf = ctypes_buf = None
    import ctypes
    ctypes_buf = ctypes.create_string_buffer(1 << 16)

    # The step as a CUDA graph, captured once after the warm-up: every replay launches the same
    # kernels on the same resident inputs, and the host enqueues one launch per step, so a delay
    # on the host (scheduling, the clock sampler) cannot open gaps inside a timed step.  The
    # replay's volumes are checked bit for bit against a direct run; --no-graph times direct calls.
    graph, graph_launches, graph_note = None, 0, "direct calls (--no-graph)"
    if not args.no_graph and side is not None:
        try:
            torch.cuda.synchronize(dev)
            ctx.lib.ds_profile_report(ctx.h, ctypes_buf, len(ctypes_buf))     # reset the launch counter
            g_ = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g_, capture_error_mode="relaxed"):
                step()
            ctx.check(ctx.lib.ds_profile_report(ctx.h, ctypes_buf, len(ctypes_buf)))
            graph_launches = int(json.loads(ctypes_buf.value.decode()).get("launches", 0))
            I_n.zero_()
            I_m.zero_()
            g_.replay()
            torch.cuda.synchronize(dev)
            rn, rm = I_n.clone(), I_m.clone()
            step()
            torch.cuda.synchronize(dev)
            if graph_launches > 0 and torch.equal(rn, I_n) and torch.equal(rm, I_m):
                graph = g_
                graph_note = "CUDA graph replay of the step (captured once; %d kernels per step; volumes " \
                             "identical to direct calls)" % graph_launches
            else:
                graph_note = "direct calls (the graph replay did not reproduce the direct volumes)"
            del rn, rm
        except Exception as e:  # capture not supported here: time direct calls
            graph_note = "direct calls (graph capture failed: %s)" % str(e).splitlines()[0][:160]
            torch.cuda.synchronize(dev)

    # timed region: K steps, per-step events on the launching stream, L2 flushed in between
    ctx.lib.ds_profile_report(ctx.h, ctypes_buf, len(ctypes_buf))     # reset counters
    ev = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(args.steps)]
    barrier(dev)
    torch.cuda.synchronize(dev)
    t_wall = time.perf_counter()
    for i in range(args.steps):
        flush.zero_()
        ev[i][0].record(stream)
        if graph is not None:
            graph.replay()
        else:
            step()
        ev[i][1].record(stream)
    torch.cuda.synchronize(dev)
    barrier(dev)
    t_wall = time.perf_counter() - t_wall
    ctx.check(ctx.lib.ds_profile_report(ctx.h, ctypes_buf, len(ctypes_buf)))
    timed_launches = int(json.loads(ctypes_buf.value.decode()).get("launches", 0))
    if graph is not None:
        timed_launches = graph_launches * args.steps
    clk = clocks.stop()
    # per-stage times from the same steps run again with the library's stage events: the events
    # sit between the kernels of a stream (no launch overlap), so they stay out of the timed region
    ctx.lib.ds_profile_enable(ctx.h, 1)
    for _ in range(min(args.steps, 20)):
        flush.zero_()
        step()
    torch.cuda.synchronize(dev)
    ctx.lib.ds_profile_enable(ctx.h, 0)
    ctx.check(ctx.lib.ds_profile_report(ctx.h, ctypes_buf, len(ctypes_buf)))
    prof = json.loads(ctypes_buf.value.decode())
    step_ms = [a.elapsed_time(b) for a, b in ev]
    total_ms = max_over_ranks(sum(step_ms), dev)
    vox_step = 2 * nvox
    value = ws * vox_step * args.steps / (total_ms / 1e3)

    # the dominant kernel timed alone as well (one stream, no overlap with the other volume)
    ctx.lib.ds_profile_report(ctx.h, ctypes_buf, len(ctypes_buf))
    ctx.lib.ds_profile_enable(ctx.h, 1)
    for _ in range(20):
        flush.zero_()
        step(single=True)
    torch.cuda.synchronize(dev)
    ctx.lib.ds_profile_enable(ctx.h, 0)
    ctx.check(ctx.lib.ds_profile_report(ctx.h, ctypes_buf, len(ctypes_buf)))
    alone = json.loads(ctypes_buf.value.decode())["stages"].get("recombine_spin", {"count": 1, "ms": float("nan")})

    # accuracy of the timed FP32 path against the FP64 path of the same kernels
    I_n64 = torch.empty(m.qgrid.count, dtype=torch.float64, device=dev)
    I_m64 = torch.empty(m.qgrid.count, dtype=torch.float64, device=dev)
    step(ds.DS_FP64, (I_n64, I_m64))
    torch.cuda.synchronize(dev)
    errs = []
    for a, b in ((I_n, I_n64), (I_m, I_m64)):
        errs.append(float((a.double() - b).abs().max() / b.abs().max()))
    # plain FP64 path throughput (a few steps)
    n64 = max(2, min(5, args.steps))
    e64 = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(n64)]
    for i in range(n64):
        flush.zero_()
        e64[i][0].record(stream)
        step(ds.DS_FP64, (I_n64, I_m64))
        e64[i][1].record(stream)
    torch.cuda.synchronize(dev)
    ms64 = sum(a.elapsed_time(b) for a, b in e64) / n64

    # end to end through the public API with host buffers (pinned), copies inside the timed
    # region: each step copies the inputs host -> device and uploads them into the models, computes
    # both volumes (one stream each, as in the device-timed steps) and copies both back to pinned
    # host memory on copy streams, so that the read-back of step i overlaps the work of step i+1
    # (device outputs double buffered; an upload waits for the previous step's kernels).
    occ_dd = torch.empty_like(occ_d)
    spin_dd = torch.empty_like(spin_d)
    dev_out = [[torch.empty(m.qgrid.count, dtype=torch.float32, device=dev) for _ in range(2)] for _ in range(2)]
    host_out = [[torch.empty(m.qgrid.count, dtype=torch.float32).pin_memory() for _ in range(2)] for _ in range(2)]
    comp_s = [torch.cuda.Stream(dev), torch.cuda.Stream(dev)]
    copy_s = [torch.cuda.Stream(dev), torch.cuda.Stream(dev)]
    comp_done = [[torch.cuda.Event() for _ in range(2)] for _ in range(2)]
    copy_done = [[torch.cuda.Event() for _ in range(2)] for _ in range(2)]
    e2e_fork = torch.cuda.Event()
    vols = ((lm_n, ds.DS_OCC, ds.DS_DIFFUSE), (lm_m, ds.DS_SPIN, ds.DS_TOTAL))

    def e2e_step(i):
        b = i % 2
        occ_dd.copy_(occ_h, non_blocking=True)
        spin_dd.copy_(spin_h, non_blocking=True)
        lm_n.upload_occupancy(occ_dd)
        lm_m.upload_spins(spin_dd)
        e2e_fork.record(stream)
        for v, (lm_, dis, mode) in enumerate(vols):
            comp_s[v].wait_event(e2e_fork)
            comp_s[v].wait_event(copy_done[b][v])       # the read-back of step i - 2 from this buffer
            with torch.cuda.stream(comp_s[v]):
                lm_.intensity(q, out=dev_out[b][v], disorder=dis, mode=mode, precision=ds.DS_FP32)
            comp_done[b][v].record(comp_s[v])
            stream.wait_event(comp_done[b][v])          # the next upload waits for these kernels
            copy_s[v].wait_event(comp_done[b][v])
            with torch.cuda.stream(copy_s[v]):
                host_out[b][v].copy_(dev_out[b][v], non_blocking=True)
            copy_done[b][v].record(copy_s[v])

    for i in range(max(3, min(5, args.warmup))):
        e2e_step(i)
    torch.cuda.synchronize(dev)
    barrier(dev)
    t0 = time.perf_counter()
    for i in range(args.steps):
        e2e_step(i)
    torch.cuda.synchronize(dev)
    e2e_s = max_over_ranks(time.perf_counter() - t0, dev)
    e2e_err = max(float((host_out[(args.steps - 1) % 2][0].to(dev) - I_n).abs().max()),
                  float((host_out[(args.steps - 1) % 2][1].to(dev) - I_m).abs().max()))
    e2e = {"value": ws * vox_step * args.steps / e2e_s, "unit": UNIT,
           "h2d_bytes_per_step": int(occ_h.numel() * occ_h.element_size() + spin_h.numel() * spin_h.element_size()),
           "d2h_bytes_per_step": int(2 * nvox * 4), "max_abs_diff_vs_device_steps": e2e_err,
           "ms_per_step": 1e3 * e2e_s / args.steps}

    # roofline of the dominant kernel, the magnetic recombination (residue-class kernel): its
    # algorithmic traffic is the intensity volume it writes (4 B per voxel) plus one read of the
    # site spectra (nsite x 3 components x n1 n2 (n3/2 + 1) complex FP32); HBM bound
    peaks, peak_src = measured_peaks()
    st = prof["stages"]
    rec = st.get("recombine_spin", {"count": 1, "ms": float("nan")})
    avg_ms = rec["ms"] / max(1, rec["count"])
    spec_bytes = NSITE * 3 * NCELL * NCELL * (NCELL // 2 + 1) * 8
    alg_bytes = nvox * 4 + spec_bytes
    achieved = alg_bytes / (avg_ms / 1e3) / 1e9
    hbm = float(peaks["hbm_gbs"])
    roofline = {"bound": "hbm", "achieved": achieved, "peak": hbm, "unit": "GB/s", "frac": achieved / hbm,
                "traffic": MAG_KERNEL_TRAFFIC, "kernel": MAG_KERNEL,
                "peak_source": "%s HBM copy bandwidth (MEASURED_PEAKS.json hbm_gbs)" % peak_src,
                "algorithmic_bytes_per_launch": alg_bytes, "avg_launch_ms": avg_ms,
                "traffic_source": MAG_KERNEL_TRAFFIC_SOURCE,
                "alone": {"avg_launch_ms": alone["ms"] / max(1, alone["count"]),
                          "achieved": alg_bytes / (alone["ms"] / max(1, alone["count"]) / 1e3) / 1e9,
                          "note": "same kernel timed on one stream without the other volume's kernels"}}
    stages = {k: {"count": v["count"], "avg_ms": v["ms"] / max(1, v["count"])} for k, v in st.items()}

    cpu = None
    if rank == 0 and ws == 1 and not args.no_cpu_baseline:
        cpu = cpu_baseline()
    serving = None
    lm_n.close()
    lm_m.close()
    ctx.close()
    rows = None
    if rank == 0 and not args.no_rows:
        rows = run_rows(dev, cpu_rows=not args.no_cpu_baseline)
    if args.serving > 0:
        serving = run_serving(args.serving, nreq_fp64=args.serving)
    line = {"metric": METRIC, "value": value, "unit": UNIT, "n_gpus": ws, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": total_ms / args.steps, "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": workload_config({"parallelism": "replicas" if ws > 1 else "single GPU",
                                       "streams": args.streams, "launch": graph_note}),
            "max_rel_err_vs_fp64": max(errs), "fp64_plain": {"ms_per_step": ms64, "value": ws * vox_step / (ms64 / 1e3)},
            "e2e": e2e, "roofline": roofline, "stages": stages, "gpu_launches": timed_launches,
            "wall_ms_per_step": 1e3 * t_wall / args.steps, "clocks": clk, "cpu_baseline": cpu,
            "serving": serving, "rows": rows}
    if rank == 0:
        print(json.dumps(line))
    return 0


# ----------------------------------------------------------------------------------------------
# the other rows of the path, each timed on its own workload (device events, warm)
# ----------------------------------------------------------------------------------------------

def device_peaks(ctx, dev):
    """FP32 / FP64 FMA and SFU throughput measured by the library's microkernels (ds_measure_peaks)."""
    import ctypes
    vals = (ctypes.c_double * 5)()
    ctx.check(ctx.lib.ds_measure_peaks(dev.index or 0, vals))
    keys = ("fp32_fma_tflops", "fp32x2_fma_tflops", "fp64_fma_tflops", "sfu_ex2_tops", "sfu_sincos_tops")
    out = {k: float(v) for k, v in zip(keys, vals)}
    out["source"] = "ds_measure_peaks: FMA-chain and SFU kernels, 8 CTAs x 256 threads per SM, this run"
    return out


def taylor_sf_flops(cells, qgrid, P, nsite):
    """Multiply-adds of the sum-factorised Taylor recombination for this grid (the kernel's own
    count, 4 flop per complex x real multiply-add): per stored k of the half spectrum and per zone
    box (the box of the grid's zones of k, and the box of the Friedel mates when it differs),
    T(P) n3 + (P+1)(P+2)/2 n2 n3 + (P+1) n1 n2 n3 per site."""
    import numpy as np
    n = list(cells)
    g0 = [int(round(qgrid.h0[a] * n[a])) for a in range(3)]
    cnt = list(qgrid.count)
    T = (P + 1) * (P + 2) * (P + 3) / 6.0
    nab = (P + 1) * (P + 2) / 2.0

    def boxes(a):
        k = np.arange(n[a] if a < 2 else n[2] // 2 + 1)
        dlo = -((-(g0[a] - k)) // n[a])
        dhi = (g0[a] + cnt[a] - 1 - k) // n[a]
        mlo = -((-(-(g0[a] + cnt[a] - 1) - k)) // n[a])
        mhi = (-g0[a] - k) // n[a]
        return dlo, np.maximum(dhi - dlo + 1, 0), mlo, np.maximum(mhi - mlo + 1, 0)

    b = [boxes(a) for a in range(3)]
    k3 = np.arange(n[2] // 2 + 1)
    has_m = (k3 >= 1) & (k3 <= n[2] - (n[2] // 2 + 1))
    work = 0.0
    for k1 in range(n[0]):
        for k2 in range(n[1]):
            d1, d2, d3 = b[0][1][k1], b[1][1][k2], b[2][1]
            m1, m2, m3 = b[0][3][k1], b[1][3][k2], b[2][3]
            wd = np.where(d1 * d2 * d3 > 0, T * d3 + nab * d2 * d3 + (P + 1) * d1 * d2 * d3, 0.0)
            wm = np.where(m1 * m2 * m3 > 0, T * m3 + nab * m2 * m3 + (P + 1) * m1 * m2 * m3, 0.0)
            same = (b[0][0][k1] == b[0][2][k1]) & (d1 == m1) & (b[1][0][k2] == b[1][2][k2]) & (d2 == m2) & \
                   (b[2][0] == b[2][2]) & (d3 == m3)
            work += float(np.sum(wd) + np.sum(np.where(has_m & ~same, wm, 0.0)))
    return 4.0 * work * nsite


def taylor_sf_adjoint_flops(cells, qgrid, P, nsite):
    """Multiply-adds of the transposed sum factorisation of the adjoint: per k of the stored half (the
    grid is symmetric about the origin) and per site, (P+1) n1 n2 n3 + (P+1)(P+2)/2 n2 n3 + T(P) n3
    over the k's box of zones, 4 flop each."""
    import numpy as np
    n = list(cells)
    g0 = [int(round(qgrid.h0[a] * n[a])) for a in range(3)]
    cnt = list(qgrid.count)
    T = (P + 1) * (P + 2) * (P + 3) / 6.0
    nab = (P + 1) * (P + 2) / 2.0
    nz = []
    for a in range(3):
        k = np.arange(n[a] if a < 2 else n[a] // 2 + 1)
        lo = -((-(g0[a] - k)) // n[a])
        hi = (g0[a] + cnt[a] - 1 - k) // n[a]
        nz.append(np.maximum(hi - lo + 1, 0).astype(np.float64))
    n1, n2, n3 = nz
    s1, s2, s3 = n1.sum(), n2.sum(), n3.sum()
    work = (P + 1) * s1 * s2 * s3 + nab * n1.size * s2 * s3 + T * n1.size * n2.size * s3
    return 4.0 * work * nsite


def fft_side_comparison(dev, nfields, cells, ours_ms, reps=3):
    """Timed side comparison, not on the path: cuFFT (through torch.fft.rfftn) on the same batch
    of real fields, materialised in HBM (the library generates the monomials inside its first
    pass instead).  Returns a dict, or the reason it could not run."""
    import torch
    try:
        x = torch.randn((nfields,) + tuple(cells), dtype=torch.float32, device=dev)
        torch.fft.rfftn(x, dim=(-3, -2, -1))
        torch.cuda.synchronize(dev)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            y = torch.fft.rfftn(x, dim=(-3, -2, -1))
        b.record()
        torch.cuda.synchronize(dev)
        ms = a.elapsed_time(b) / reps
        nbytes = x.numel() * 4 + y.numel() * 8
        del x, y
        torch.cuda.empty_cache()
        return {"library": "cuFFT via torch.fft.rfftn (forward, R2C, FP32)", "fields": nfields,
                "cells": list(cells), "ms": ms, "library_GBps": nbytes / (ms / 1e3) / 1e9,
                "ours_ms": ours_ms,
                "note": "side comparison only; the library's FFT stage also generates the monomial fields"}
    except Exception as e:  # the comparison must never stop the bench
        return {"unavailable": "%s: %s" % (type(e).__name__, str(e)[:200])}


def run_rows(dev, cpu_rows=True):
    """One measurement per remaining step of the path: the Taylor (displacive) recombination and
    its adjoint on the fcc 32^3 / 321^3 case, Lanczos resampling on a 1025^3 volume, exact sub-box
    averaging and arbitrary-wavevector resampling on an (h h l) plane of 401 x 401 points."""
    import ctypes
    import numpy as np
    import torch
    import paper_1809_07088_gb300 as ds
    import synthetic as syn

    peaks, _ = measured_peaks()
    hbm = float(peaks["hbm_gbs"])
    ctx = ds.Context(dev.index or 0)
    buf = ctypes.create_string_buffer(1 << 16)
    alu = device_peaks(ctx, dev)
    fp32 = max(alu["fp32_fma_tflops"], alu["fp32x2_fma_tflops"])   # the faster FP32 FMA form

    def timed(fn, reps=3):
        fn()
        torch.cuda.synchronize(dev)
        ctx.lib.ds_profile_report(ctx.h, buf, len(buf))
        ctx.lib.ds_profile_enable(ctx.h, 1)
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            fn()
        b.record()
        torch.cuda.synchronize(dev)
        ctx.lib.ds_profile_enable(ctx.h, 0)
        ctx.check(ctx.lib.ds_profile_report(ctx.h, buf, len(buf)))
        st = json.loads(buf.value.decode())["stages"]
        return a.elapsed_time(b) / reps, {k: v["ms"] / max(1, v["count"]) for k, v in st.items()}

    rows = {"alu_peaks": alu}
    # Taylor recombination (S1-S5 displacive) and adjoint (S7): fcc 32^3, 321^3 voxels, eps 1e-8
    m = syn.displacive_fcc(cells=(32, 32, 32), sigma=0.1, seed=5)
    m.qgrid = syn.symmetric_qgrid(5.0, m.cells)
    lm = ds.Model(ctx, m.lattice, m.sites, m.cells, 1, m.scat_len, m.ff_kind, m.ff_coef)
    lm.upload_displacements(np.ascontiguousarray(m.disp))
    q = (m.qgrid.h0, m.qgrid.step, m.qgrid.count)
    out = torch.empty(m.qgrid.count, dtype=torch.float32, device=dev)
    for zonal in (0, 1):
        o = dict(disorder=ds.DS_DISP, mode=ds.DS_TOTAL, precision=ds.DS_FP32, taylor_order=-1, taylor_eps=1e-8,
                 taylor_zonal=zonal)
        _, info = lm.intensity(q, out=out, **o)
        ms, st = timed(lambda: lm.intensity(q, out=out, **o))
        T = info["n_monomials"]
        rec = st.get("recombine_disp", float("nan"))
        row = {"workload": "fcc 32^3 cells, u ~ N(0, 0.1^2), |hkl| <= 5 step 1/32 (321^3 voxels), FP32, eps 1e-8",
               "taylor_order": info["taylor_order"], "monomials": T, "ms": ms, "stages_ms": st,
               "voxels_per_s": m.qgrid.nvox / (ms / 1e3)}
        if zonal == 0:
            flops = taylor_sf_flops(m.cells, m.qgrid, info["taylor_order"], m.nsite)
            row["kernel"] = "k_taylor_sf (sum factorisation)"
            row["roofline"] = {"bound": "alu", "achieved": flops / (rec / 1e3) / 1e12, "peak": fp32,
                               "unit": "TFLOP/s", "frac": flops / (rec / 1e3) / 1e12 / fp32,
                               "note": "Horner multiply-adds of the three axis contractions over each k's "
                                       "zones (complex x real = 4 flop), peak measured in this run"}
        else:
            row["kernel"] = "k_recomb_disp (per-zone orders, per voxel)"
        rows["taylor_fcc32_zonal%d" % zonal] = row
    dL = torch.ones(m.qgrid.count, dtype=torch.float32, device=dev)
    g = torch.empty((1, m.nsite) + tuple(m.cells) + (3,), dtype=torch.float32, device=dev)
    ms, st = timed(lambda: lm.backward(q, dL, grad=g, disorder=ds.DS_DISP, mode=ds.DS_TOTAL, precision=ds.DS_FP32,
                                       taylor_order=-1, taylor_eps=1e-8), reps=2)
    az = st.get("adjoint_z", float("nan"))
    aflops = taylor_sf_adjoint_flops(m.cells, m.qgrid, rows["taylor_fcc32_zonal0"]["taylor_order"], m.nsite)
    rows["adjoint_fcc32"] = {"workload": "dchi2/du of the fcc 32^3 case above, FP32", "ms": ms, "stages_ms": st,
                             "kernel": "k_adj_taylor_sf (transposed sum factorisation)",
                             "roofline": {"bound": "alu", "achieved": aflops / (az / 1e3) / 1e12, "peak": fp32,
                                          "unit": "TFLOP/s", "frac": aflops / (az / 1e3) / 1e12 / fp32,
                                          "note": "multiply-adds of the three power sums over each k's zones "
                                                  "(complex x real = 4 flop), peak measured in this run"}}
    # side comparison only (not on the path): the library FFT of the same batch of fields
    nf_fcc = m.nsite * rows["taylor_fcc32_zonal0"]["monomials"]
    rows["fft_side_comparison"] = fft_side_comparison(dev, nf_fcc, m.cells,
                                                      rows["taylor_fcc32_zonal0"]["stages_ms"].get("fft"))
    lm.close()
    del out, dL, g

    # Lanczos resampling (S6a): 1025^3 voxels (|hkl| <= 8 step 1/64), m = 2, m' = 8, occupancy
    n = 64
    mo = syn.Model(lattice=(4.0, 4.0, 4.0, 90.0, 90.0, 90.0), sites=np.array([[0.0, 0.0, 0.0]]),
                   scat_len=np.ones(1), ff_kind=np.zeros(1, dtype=np.int32), ff_coef=np.zeros((1, 9)),
                   cells=(n, n, n), nmodels=1)
    mo.occ = (np.random.default_rng(3).random((1, 1, n, n, n)) < 0.5).astype(np.uint8)
    lo = ds.Model(ctx, mo.lattice, mo.sites, mo.cells, 1, mo.scat_len, mo.ff_kind, mo.ff_coef)
    lo.upload_occupancy(np.ascontiguousarray(mo.occ))
    qg = syn.symmetric_qgrid(8.0, mo.cells)
    q = (qg.h0, qg.step, qg.count)
    out = torch.empty(qg.count, dtype=torch.float32, device=dev)
    ms, st = timed(lambda: lo.intensity(q, out=out, disorder=ds.DS_OCC, mode=ds.DS_DIFFUSE, precision=ds.DS_FP32,
                                        smoothing=ds.DS_SMOOTH_LANCZOS, lanczos_m=2, lanczos_mprime=8), reps=2)
    lz = st.get("lanczos", float("nan"))
    h = 7
    ext = [c + 2 * h for c in qg.count]
    c = qg.count
    # two passes: axes 2 and 1 fused (read the halo-extended volume, write [ext0][c1][c2]), then
    # axis 0 (read that, write the output)
    lz_bytes = 4.0 * (ext[0] * ext[1] * ext[2] + 2 * ext[0] * c[1] * c[2] + c[0] * c[1] * c[2])
    rows["lanczos_1025cubed"] = {
        "workload": "occupancy 64^3 cells, |hkl| <= 8 step 1/64 (1025^3 voxels), Lanczos m = 2, m' = 8, FP32",
        "ms": ms, "stages_ms": st,
        "roofline": {"bound": "hbm", "achieved": lz_bytes / (lz / 1e3) / 1e9, "peak": hbm, "unit": "GB/s",
                     "frac": lz_bytes / (lz / 1e3) / 1e9 / hbm,
                     "note": "two passes (in-plane axes fused, then the outer axis), each reading and writing "
                             "its volume once (4 B per voxel)"}}
    lo.close()
    del out

    # exact sub-box averaging (S6b) and arbitrary wavevectors (S6a'): the pyrochlore workload
    mp = syn.pyrochlore_occ_mag()
    lp = ds.Model(ctx, mp.lattice, mp.sites, mp.cells, 1, mp.scat_len, mp.ff_kind, mp.ff_coef)
    lp.upload_occupancy(np.ascontiguousarray(mp.occ))
    q = (mp.qgrid.h0, mp.qgrid.step, mp.qgrid.count)
    out = torch.empty(mp.qgrid.count, dtype=torch.float32, device=dev)
    ms, st = timed(lambda: lp.intensity(q, out=out, disorder=ds.DS_OCC, mode=ds.DS_DIFFUSE, precision=ds.DS_FP32,
                                        smoothing=ds.DS_SMOOTH_SUBBOX, subbox_n=5), reps=2)
    rows["subbox_pyrochlore"] = {"workload": "pyrochlore occupancy 20^3, 241^3 voxels, n_sb = 5, FP32", "ms": ms,
                                 "stages_ms": st, "voxels_per_s": mp.qgrid.nvox / (ms / 1e3)}
    u, v = np.meshgrid(np.linspace(-6.0, 6.0, 401), np.linspace(-6.0 * 2 ** 0.5, 6.0 * 2 ** 0.5, 401), indexing="ij")
    hkl = torch.from_numpy(np.stack([u.ravel(), u.ravel(), v.ravel()], axis=1)).to(dev)
    pts = torch.empty(hkl.shape[0], dtype=torch.float32, device=dev)
    ms, st = timed(lambda: lp.intensity_points(hkl, out=pts, disorder=ds.DS_OCC, mode=ds.DS_DIFFUSE,
                                               precision=ds.DS_FP32, lanczos_m=2, lanczos_mprime=2), reps=2)
    rows["points_hhl_plane"] = {"workload": "(h h l) plane 401 x 401 points, |h| <= 6, |l| <= 6 sqrt 2, pyrochlore "
                                            "occupancy 20^3, Lanczos m = 2, FP32 (the paper's plane geometry)",
                                "ms": ms, "stages_ms": st, "points_per_s": hkl.shape[0] / (ms / 1e3)}
    lp.close()

    # sub-boxes by direct summation (S6b'): random origins covering the fcc 32^3 displacive
    # supercell, n_sb = 5, exact exp(i Q.u), (h h l) plane 201 x 201, DIFFUSE
    md = syn.displacive_fcc(cells=(32, 32, 32), sigma=0.1, seed=5)
    ld = ds.Model(ctx, md.lattice, md.sites, md.cells, 1, md.scat_len, md.ff_kind, md.ff_coef)
    ld.upload_displacements(np.ascontiguousarray(md.disp))
    org = syn.covering_origins(np.random.default_rng(7), 1, md.cells, 5)
    u, v = np.meshgrid(np.linspace(-5.0, 5.0, 201), np.linspace(-5.0, 5.0, 201), indexing="ij")
    hkl = torch.from_numpy(np.stack([u.ravel(), u.ravel(), v.ravel()], axis=1)).to(dev)
    pts = torch.empty(hkl.shape[0], dtype=torch.float32, device=dev)
    ms, st = timed(lambda: ld.subbox_points(hkl, org, out=pts, disorder=ds.DS_DISP, mode=ds.DS_DIFFUSE,
                                            precision=ds.DS_FP32, subbox_n=5), reps=2)
    terms = float(hkl.shape[0]) * md.natom      # one per atom and point: the cells are shared by the boxes
    sb = st.get("subbox_cells", float("nan"))
    mufu = alu["sfu_sincos_tops"] * 1e12   # (sin, cos) pairs per second, measured in this run
    rows["subbox_random_disp_fcc32_plane"] = {
        "workload": "fcc 32^3 displacive (u ~ N(0, 0.1^2)), %d random origins covering every cell, n_sb = 5, "
                    "(h h l) plane 201 x 201 |h|, |l| <= 5, DIFFUSE, FP32" % org.shape[0],
        "ms": ms, "stages_ms": st, "points_per_s": hkl.shape[0] / (ms / 1e3),
        "roofline": {"bound": "alu", "achieved": terms / (sb / 1e3) / 1e12, "peak": mufu / 1e12,
                     "unit": "Tterm/s", "frac": terms / (sb / 1e3) / mufu,
                     "note": "one exp(i Q.u) (one SFU sine-cosine pair) per atom and point, cell amplitudes shared "
                             "by the boxes; peak: __sincosf pairs per second measured in this run"}}
    ld.close()

    # magnetic + displacive coupling through T_mu(G) (Eq. mag_sf): pyrochlore 20^3, |hkl| <= 2
    mm = syn.pyrochlore_mag_disp(cells=(20, 20, 20), hmax=2.0)
    lmg = ds.Model(ctx, mm.lattice, mm.sites, mm.cells, 1, mm.scat_len, mm.ff_kind, mm.ff_coef)
    lmg.upload_spins(np.ascontiguousarray(mm.spins))
    lmg.upload_displacements(np.ascontiguousarray(mm.disp))
    q = (mm.qgrid.h0, mm.qgrid.step, mm.qgrid.count)
    out = torch.empty(mm.qgrid.count, dtype=torch.float32, device=dev)
    ms, st = timed(lambda: lmg.intensity(q, out=out, disorder=ds.DS_SPIN, mode=ds.DS_TOTAL, precision=ds.DS_FP32,
                                         dw_coupling=1), reps=2)
    dwms = st.get("debye_waller", float("nan"))
    dwb = 4.0 * mm.qgrid.nvox * mm.nsite + 12.0 * mm.natom   # factors written, displacements read
    rows["mag_dw_pyrochlore20"] = {
        "workload": "magnetic pyrochlore 20^3 with u ~ N(0, 0.05^2), |hkl| <= 2 step 1/20 (%d^3 voxels), "
                    "T_mu(G) per voxel and site, FP32" % mm.qgrid.count[0],
        "ms": ms, "stages_ms": st, "voxels_per_s": mm.qgrid.nvox / (ms / 1e3),
        "roofline": {"bound": "hbm", "achieved": dwb / (dwms / 1e3) / 1e9, "peak": hbm, "unit": "GB/s",
                     "frac": dwb / (dwms / 1e3) / 1e9 / hbm,
                     "note": "T_mu(G) from the moments of the displacements: factors written plus displacements "
                             "read; five kernels, launch and FP64 latency at this size"}}
    lmg.close()

    # the displacive fcc 8^3 workload, plain FP64 (Taylor order by the remainder bound at eps 1e-8),
    # whole 64^3 volume; CPU: the oracle's direct sum of the whole volume on every host core
    m1 = syn.displacive_fcc()
    l1 = ds.Model(ctx, m1.lattice, m1.sites, m1.cells, 1, m1.scat_len, m1.ff_kind, m1.ff_coef)
    l1.upload_displacements(np.ascontiguousarray(m1.disp))
    q = (m1.qgrid.h0, m1.qgrid.step, m1.qgrid.count)
    out = torch.empty(m1.qgrid.count, dtype=torch.float64, device=dev)
    o1 = dict(disorder=ds.DS_DISP, mode=ds.DS_DIFFUSE, precision=ds.DS_FP64, taylor_order=-1, taylor_eps=1e-8)
    _, info = l1.intensity(q, out=out, **o1)
    ms, st = timed(lambda: l1.intensity(q, out=out, **o1))
    row = {"workload": "fcc 8^3 cells (2048 atoms), u ~ N(0, 0.1^2), h,k,l in [-4, 4) step 1/8 (64^3 voxels), "
                       "DIFFUSE, plain FP64, eps 1e-8",
           "taylor_order": info["taylor_order"], "x_max": info["x_max"], "monomials": info["n_monomials"],
           "ms": ms, "stages_ms": st, "voxels_per_s": m1.qgrid.nvox / (ms / 1e3)}
    if cpu_rows:
        rate, dt, thr = cpu_direct_rate(m1, m1.qgrid.hkl(), 1)
        row["cpu_baseline"] = {"value": rate, "unit": UNIT, "cores": thr, "kind": "oracle",
                               "sample": "the whole 64^3 volume by the direct sum (C, OpenMP), %.1f s" % dt}
    rows["c1_fcc8_fp64"] = row
    l1.close()
    del out

    # the large displacive workload: perovskite 64^3 (1.31 M atoms), 1025^3 voxels, FP32 at eps 1e-5,
    # and the FP32 path against the plain FP64 path on the two |Q|-maximal corner zones and the centre
    # zone (same order); CPU: the oracle's direct sum on sampled voxels of those zones
    m3 = syn.perovskite_correlated()
    l3 = ds.Model(ctx, m3.lattice, m3.sites, m3.cells, 1, m3.scat_len, m3.ff_kind, m3.ff_coef)
    l3.upload_displacements(np.ascontiguousarray(m3.disp))
    q = (m3.qgrid.h0, m3.qgrid.step, m3.qgrid.count)
    out = torch.empty(m3.qgrid.count, dtype=torch.float32, device=dev)
    o3 = dict(disorder=ds.DS_DISP, mode=ds.DS_DIFFUSE, precision=ds.DS_FP32, taylor_order=-1, taylor_eps=1e-5,
              smoothing=ds.DS_SMOOTH_LANCZOS, lanczos_m=2, lanczos_mprime=8)
    _, info = l3.intensity(q, out=out, **o3)
    ms, st = timed(lambda: l3.intensity(q, out=out, **o3), reps=2)
    P = info["taylor_order"]
    del out
    torch.cuda.empty_cache()
    n = m3.cells[0]
    zerr, zpeak = [], 0.0
    for H in ((7, 7, 7), (-8, -8, -8), (0, 0, 0)):
        zq = (tuple(float(h) for h in H), (1.0 / n,) * 3, (n, n, n))
        z32 = torch.empty((n, n, n), dtype=torch.float32, device=dev)
        z64 = torch.empty((n, n, n), dtype=torch.float64, device=dev)
        l3.intensity(zq, out=z32, disorder=ds.DS_DISP, mode=ds.DS_DIFFUSE, precision=ds.DS_FP32, taylor_order=P)
        l3.intensity(zq, out=z64, disorder=ds.DS_DISP, mode=ds.DS_DIFFUSE, precision=ds.DS_FP64, taylor_order=P)
        torch.cuda.synchronize(dev)
        zerr.append(float((z32.double() - z64).abs().max()))
        zpeak = max(zpeak, float(z64.abs().max()))
        del z32, z64
    rec = st.get("recombine_disp", float("nan"))
    flops = taylor_sf_flops(m3.cells, m3.qgrid, P, m3.nsite)
    row = {"workload": "perovskite 64^3 cells (1,310,720 atoms), correlated u (0.08 A rms), 4-Gaussian form "
                       "factors, |hkl| <= 8 step 1/64 (1025^3 voxels), DIFFUSE, FP32, eps 1e-5, Lanczos m = 2, "
                       "m' = 8 (I(G) on the 1039^3 halo-extended grid, then the two resampling passes)",
           "taylor_order": P, "x_max": info["x_max"], "monomials": info["n_monomials"], "ms": ms, "stages_ms": st,
           "voxels_per_s": m3.qgrid.nvox / (ms / 1e3),
           "max_rel_err_vs_fp64_corner_zones": max(zerr) / zpeak,
           "zones_checked": "H = (7,7,7), (-8,-8,-8), (0,0,0): every voxel of the unsmoothed volume, FP32 against the plain FP64 path",
           "kernel": "k_taylor_sf (sum factorisation)",
           "roofline": {"bound": "alu", "achieved": flops / (rec / 1e3) / 1e12, "peak": fp32, "unit": "TFLOP/s",
                        "frac": flops / (rec / 1e3) / 1e12 / fp32,
                        "note": "Horner multiply-adds of the three axis contractions over each k's zones "
                                "(complex x real = 4 flop), peak measured in this run"}}
    if cpu_rows:
        rng = np.random.default_rng(5)
        G = np.concatenate([np.asarray(H)[None, :] * n + rng.integers(0, n, (24, 3))
                            for H in ((7, 7, 7), (-8, -8, -8), (0, 0, 0))])
        rate, dt, thr = cpu_direct_rate(m3, G / float(n), 1)
        row["cpu_baseline"] = {"value": rate, "unit": UNIT, "cores": thr, "kind": "oracle",
                               "sample": "72 voxels of the corner and centre zones by the direct sum over all "
                                         "1.31 M atoms (C, OpenMP), %.1f s, voxels/s extrapolated" % dt}
    rows["c3_perovskite64"] = row
    l3.close()
    torch.cuda.empty_cache()
    ctx.close()
    return rows


def run_profile_workload(name):
    """A small case of one row, run twice, for ncu captures (a few hundred MB on the device):
    taylor = fcc 32^3, 321^3 voxels, P = 12 (taylor30: P = 30, 5456 monomials); fft64 = the perovskite 64^3 model at P = 4 (175 fields
    of 64^3), |hkl| <= 2; lanczos = occupancy 32^3 cells, 513^3 voxels,
    m = 2, m' = 8 (lanczos1025: the full 64^3-cell, 1025^3-voxel row, about 13 GB on the device:
    for one-pass launch lists only); subbox = the pyrochlore occupancy volume with n_sb = 5; subbox_dft = the
    random-origin displacive boxes on a 101 x 101 (h h l) plane; dw = the magnetic pyrochlore
    with T_mu(G), |hkl| <= 1."""
    import ctypes
    import numpy as np
    import torch
    import paper_1809_07088_gb300 as ds
    import synthetic as syn
    ctx = ds.Context(0)
    if name in ("taylor", "taylor30"):
        m = syn.displacive_fcc(cells=(32, 32, 32), sigma=0.1, seed=5)
        m.qgrid = syn.symmetric_qgrid(5.0, m.cells)
        lm = ds.Model(ctx, m.lattice, m.sites, m.cells, 1, m.scat_len, m.ff_kind, m.ff_coef)
        lm.upload_displacements(np.ascontiguousarray(m.disp))
        opts = dict(disorder=ds.DS_DISP, mode=ds.DS_TOTAL, precision=ds.DS_FP32,
                    taylor_order=12 if name == "taylor" else 30)
    elif name == "fft64":
        # the perovskite 64^3 model at Taylor order 4: 5 sites x 35 monomials = 175 fields of 64^3
        m = syn.perovskite_correlated()
        m.qgrid = syn.symmetric_qgrid(2.0, m.cells)
        lm = ds.Model(ctx, m.lattice, m.sites, m.cells, 1, m.scat_len, m.ff_kind, m.ff_coef)
        lm.upload_displacements(np.ascontiguousarray(m.disp))
        opts = dict(disorder=ds.DS_DISP, mode=ds.DS_TOTAL, precision=ds.DS_FP32, taylor_order=4)
    elif name in ("lanczos", "lanczos1025"):
        n = 64 if name == "lanczos1025" else 32
        m = syn.Model(lattice=(4.0, 4.0, 4.0, 90.0, 90.0, 90.0), sites=np.array([[0.0, 0.0, 0.0]]),
                      scat_len=np.ones(1), ff_kind=np.zeros(1, dtype=np.int32), ff_coef=np.zeros((1, 9)),
                      cells=(n, n, n), nmodels=1)
        m.occ = (np.random.default_rng(3).random((1, 1, n, n, n)) < 0.5).astype(np.uint8)
        m.qgrid = syn.symmetric_qgrid(8.0, m.cells)
        lm = ds.Model(ctx, m.lattice, m.sites, m.cells, 1, m.scat_len, m.ff_kind, m.ff_coef)
        lm.upload_occupancy(np.ascontiguousarray(m.occ))
        opts = dict(disorder=ds.DS_OCC, mode=ds.DS_DIFFUSE, precision=ds.DS_FP32, smoothing=ds.DS_SMOOTH_LANCZOS,
                    lanczos_m=2, lanczos_mprime=8)
    elif name == "subbox_dft":
        m = syn.displacive_fcc(cells=(32, 32, 32), sigma=0.1, seed=5)
        lm = ds.Model(ctx, m.lattice, m.sites, m.cells, 1, m.scat_len, m.ff_kind, m.ff_coef)
        lm.upload_displacements(np.ascontiguousarray(m.disp))
        org = syn.covering_origins(np.random.default_rng(7), 1, m.cells, 5)
        u, v = np.meshgrid(np.linspace(-5.0, 5.0, 101), np.linspace(-5.0, 5.0, 101), indexing="ij")
        hkl = torch.from_numpy(np.stack([u.ravel(), u.ravel(), v.ravel()], axis=1)).cuda()
        pts = torch.empty(hkl.shape[0], dtype=torch.float32, device="cuda")
        opts = dict(disorder=ds.DS_DISP, mode=ds.DS_DIFFUSE, precision=ds.DS_FP32, subbox_n=5)
        call = lambda: lm.subbox_points(hkl, org, out=pts, **opts)
    elif name == "dw":
        m = syn.pyrochlore_mag_disp(cells=(20, 20, 20), hmax=1.0)
        lm = ds.Model(ctx, m.lattice, m.sites, m.cells, 1, m.scat_len, m.ff_kind, m.ff_coef)
        lm.upload_spins(np.ascontiguousarray(m.spins))
        lm.upload_displacements(np.ascontiguousarray(m.disp))
        opts = dict(disorder=ds.DS_SPIN, mode=ds.DS_TOTAL, precision=ds.DS_FP32, dw_coupling=1)
    else:
        m = syn.pyrochlore_occ_mag()
        lm = ds.Model(ctx, m.lattice, m.sites, m.cells, 1, m.scat_len, m.ff_kind, m.ff_coef)
        lm.upload_occupancy(np.ascontiguousarray(m.occ))
        opts = dict(disorder=ds.DS_OCC, mode=ds.DS_DIFFUSE, precision=ds.DS_FP32, smoothing=ds.DS_SMOOTH_SUBBOX,
                    subbox_n=5)
    if name != "subbox_dft":
        q = (m.qgrid.h0, m.qgrid.step, m.qgrid.count)
        out = torch.empty(m.qgrid.count, dtype=torch.float32, device="cuda")
        call = lambda: lm.intensity(q, out=out, **opts)
    call()
    torch.cuda.synchronize()
    buf = ctypes.create_string_buffer(1 << 16)
    ctx.lib.ds_profile_report(ctx.h, buf, len(buf))
    ctx.lib.ds_profile_enable(ctx.h, 1)
    call()
    torch.cuda.synchronize()
    ctx.check(ctx.lib.ds_profile_report(ctx.h, buf, len(buf)))
    print(json.dumps({"profile_workload": name, "stages": json.loads(buf.value.decode())["stages"]}))
    lm.close()
    ctx.close()
    return 0


# ----------------------------------------------------------------------------------------------
# serving: Poisson arrivals of mixed requests through ds_submit / ds_wait
# ----------------------------------------------------------------------------------------------

SERVE_SIZES = (16, 32, 48, 64)
SERVE_NSITE = (1, 2, 4, 8, 16)


def _serving_pool(ds, ctx, syn):
    """Resident models: supercells 16^3..64^3 x {occupancy, spin, displacement} x nsite buckets."""
    import numpy as np
    pool = {}
    for n in SERVE_SIZES:
        for kind in (0, 1, 2):
            for ns in SERVE_NSITE:
                spec = dict(n=n, kind=kind, nsite=ns, seed=1000 * n + 100 * kind + ns, hmax=4.0)
                m = syn.serving_model(spec)
                lm = ds.Model(ctx, m.lattice, m.sites, m.cells, 1, m.scat_len, m.ff_kind, m.ff_coef)
                if m.occ is not None:
                    lm.upload_occupancy(np.ascontiguousarray(m.occ))
                if m.spins is not None:
                    lm.upload_spins(np.ascontiguousarray(m.spins))
                if m.disp is not None:
                    lm.upload_displacements(np.ascontiguousarray(m.disp))
                pool[(n, kind, ns)] = (lm, m)
    return pool


def _bucket(nsite):
    return min(SERVE_NSITE, key=lambda b: (abs(b - nsite), b))


def _serve_stream(ds, ctx, pool, reqs, precision, rate_hz, seed, svc=None):
    """Replay `reqs` with Poisson arrivals at rate_hz; returns latency percentiles and, given the
    service time of each request type alone (`svc`), the slowdown percentiles (latency / service
    time: how much queueing and sharing stretched each request, independent of its size)."""
    import numpy as np
    import threading
    import torch
    rng = np.random.default_rng(seed)
    arrivals = np.cumsum(rng.exponential(1.0 / rate_hz, len(reqs)))
    dt = torch.float64 if precision == 0 else torch.float32
    pending = []
    lock = threading.Lock()
    cond = threading.Condition(lock)
    done = {"n": 0}
    results = []

    def submitter():
        t0 = time.perf_counter()
        for t_arr, r in zip(arrivals, reqs):
            lm, m = pool[(r["n"], r["kind"], _bucket(r["nsite"]))]
            delay = t0 + t_arr - time.perf_counter()
            if delay > 0:
                time.sleep(delay)
            out = torch.empty(m.qgrid.count, dtype=dt, device="cuda")
            opts = dict(disorder=r["kind"], mode=1 if r["kind"] != 1 else 0, precision=precision)
            if r["kind"] == 2:
                opts.update(taylor_order=-1, taylor_eps=1e-6)
            tk = lm.submit((m.qgrid.h0, m.qgrid.step, m.qgrid.count), out, **opts)
            with cond:
                pending.append((tk, out, m.qgrid.nvox, (r["n"], r["kind"], _bucket(r["nsite"]))))
                cond.notify()

    th = threading.Thread(target=submitter)
    t_start = time.perf_counter()
    th.start()
    got = 0
    while got < len(reqs):
        with cond:
            while not pending:
                cond.wait(1.0)
            tk, out, nvox, key = pending.pop(0)
        info = ctx.wait(tk, 600.0)
        results.append((info.latency_ms, info.gpu_ms, nvox, key))
        del out
        got += 1
    th.join()
    makespan = time.perf_counter() - t_start
    lat = np.array([r[0] for r in results])
    vox = sum(r[2] for r in results)
    res = {"requests": len(reqs), "rate_hz": rate_hz, "p50_ms": float(np.percentile(lat, 50)),
           "p99_ms": float(np.percentile(lat, 99)), "mean_ms": float(lat.mean()),
           "p99_over_p50": float(np.percentile(lat, 99) / np.percentile(lat, 50)),
           "throughput": vox / makespan, "unit": UNIT, "makespan_s": makespan}
    if svc:
        sd = np.array([r[0] / (1e3 * svc[r[3]]) for r in results])
        res.update({"slowdown_p50": float(np.percentile(sd, 50)), "slowdown_p99": float(np.percentile(sd, 99)),
                    "slowdown_p99_over_p50": float(np.percentile(sd, 99) / np.percentile(sd, 50)),
                    "service_ms_min_max": [1e3 * min(svc.values()), 1e3 * max(svc.values())]})
    return res


def run_serving(nreq, nreq_fp64=32, seed=4):
    """Mixed-request serving: calibrate the service time of each pool entry, then replay a
    Poisson stream at ~70% utilisation (FP32), and the same requests on the plain FP64 path (its own
    70% rate)."""
    import numpy as np
    import torch
    import paper_1809_07088_gb300 as ds
    import synthetic as syn
    torch.cuda.set_device(0)
    ctx = ds.Context(0, hbm_budget=64 << 30)
    pool = _serving_pool(ds, ctx, syn)
    reqs = syn.serving_mix(nreq=nreq, seed=seed)
    out = {}
    for precision, n in ((1, nreq), (0, nreq_fp64)):
        # service time of each request type alone (warm, sequential)
        svc = {}
        sub = reqs[:n]
        used = {(r["n"], r["kind"], _bucket(r["nsite"])) for r in sub}
        for key, (lm, m) in pool.items():
            if key not in used:
                continue
            o = torch.empty(m.qgrid.count, dtype=torch.float64 if precision == 0 else torch.float32, device="cuda")
            opts = dict(disorder=key[1], mode=1 if key[1] != 1 else 0, precision=precision)
            if key[1] == 2:
                opts.update(taylor_order=-1, taylor_eps=1e-6)
            lm.intensity((m.qgrid.h0, m.qgrid.step, m.qgrid.count), out=o, **opts)
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            lm.intensity((m.qgrid.h0, m.qgrid.step, m.qgrid.count), out=o, **opts)
            torch.cuda.synchronize()
            svc[key] = time.perf_counter() - t0
            del o
        mean_svc = float(np.mean([svc[(r["n"], r["kind"], _bucket(r["nsite"]))] for r in sub]))
        rate = 0.7 / mean_svc
        out["fp32" if precision == 1 else "fp64_plain"] = _serve_stream(ds, ctx, pool, sub, precision, rate, seed, svc)
        out["fp32" if precision == 1 else "fp64_plain"]["mean_service_ms"] = 1e3 * mean_svc
    for lm, _ in pool.values():
        lm.close()
    ctx.close()
    return out


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=1000)
    ap.add_argument("--warmup", type=int, default=10)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--serving", type=int, default=512, help="requests in the serving stream (0 = skip)")
    ap.add_argument("--no-rows", action="store_true", help="skip the per-row measurements")
    ap.add_argument("--no-graph", action="store_true", help="time direct calls instead of a replayed CUDA graph")
    ap.add_argument("--profile-workload", choices=["taylor", "taylor30", "fft64", "lanczos", "lanczos1025", "subbox", "subbox_dft", "dw"], default=None,
                    help="run one small row workload twice (for ncu captures) and exit")
    ap.add_argument("--streams", type=int, default=2, choices=[1, 2],
                    help="2: the two volumes of a step on two streams (their kernels overlap)")
    args = ap.parse_args()
    if args.warmup < 3:
        args.warmup = 3
    if args.profile_workload:
        return run_profile_workload(args.profile_workload)
    if args.impl == "reference":
        return run_reference(args)
    return run_ours(args)


if __name__ == "__main__":
    sys.exit(main())
