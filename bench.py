"""Throughput of the first-level J/psi event selection on GB300.

One step = one pass of the whole hot path over one batch: the counting pass
(triplet formation, fit and cut, chaining, accept bits), the scan of per-unit
counts and the triplet-writing pass, i.e. a jpsi_run call.  The default batch
is the 10^6-event Poisson(100) workload (4 stations x 3 layers, ~1 200 hits
per event, 14.4 GB of FP32 hits, far larger than L2), synthetic and seeded.

  python bench.py [--gpus N --steps K --warmup W] [--impl reference]

Prints one JSON line (rank 0).  Under torchrun each rank processes its own
10^6 events (weak scaling, no collective on the data path).
"""
from __future__ import annotations

import argparse
import hashlib
import re
import json
import os
import statistics
import subprocess
import sys
import tempfile
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
sys.path.insert(0, ROOT)

METRIC = "events/s on 1 GB300 (bit-exact accept bits), batched vs plain; p50/p99 latency"
UNIT = "events/s"


def shard(rank, n_per_rank):
    """Events of one rank under torchrun: each rank owns its own contiguous
    range of the workload's event stream (weak scaling, no data exchange)."""
    return rank * n_per_rank, n_per_rank


def max_over_ranks(value, dist):
    """The slowest rank's time (the job's time): all-reduce MAX over gloo."""
    import torch
    t = torch.tensor([float(value)], dtype=torch.float64)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t[0])


def dist_info():
    rank = int(os.environ.get("RANK", "0"))
    world = int(os.environ.get("WORLD_SIZE", "1"))
    local = int(os.environ.get("LOCAL_RANK", "0"))
    return rank, world, local


class Clocks:
    """nvidia-smi sampling of SM clocks and throttle reasons during a region."""

    Q = ("index,clocks.sm,clocks.max.sm,power.draw,clocks_event_reasons.active,clocks_event_reasons.hw_slowdown,"
         "clocks_event_reasons.hw_thermal_slowdown,clocks_event_reasons.sw_thermal_slowdown,"
         "clocks_event_reasons.sw_power_cap")

    def __init__(self, gpu):
        self.gpu = gpu
        self.proc = None
        self.path = None

    def start(self):
        fd, self.path = tempfile.mkstemp(prefix="clocks", suffix=".csv")
        os.close(fd)
        try:
            self.proc = subprocess.Popen(["nvidia-smi", "-i", str(self.gpu), f"--query-gpu={self.Q}",
                                          "--format=csv,noheader,nounits", "-lms", "200"],
                                         stdout=open(self.path, "w"), stderr=subprocess.DEVNULL)
        except OSError:
            self.proc = None

    def stop(self):
        if self.proc is None:
            return {"sm_mhz": None, "sm_max_mhz": None, "reasons": ["nvidia-smi unavailable"]}
        time.sleep(0.25)
        self.proc.terminate()
        self.proc.wait()
        sm, mx, reasons = [], [], set()
        names = ["hw_slowdown", "hw_thermal_slowdown", "sw_thermal_slowdown", "sw_power_cap"]
        for line in open(self.path):
            f = [v.strip() for v in line.split(",")]
            if len(f) < 9:
                continue
            try:
                sm.append(float(f[1]))
                mx.append(float(f[2]))
            except ValueError:
                continue
            for n, v in zip(names, f[5:9]):
                if v.lower().startswith("active"):
                    reasons.add(n)
        os.unlink(self.path)
        return {"sm_mhz": statistics.median(sm) if sm else None, "sm_max_mhz": max(mx) if mx else None,
                "reasons": sorted(reasons), "samples": len(sm)}


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        d = json.load(open(p))
        return float(d["hbm_gbs"]), "measured"
    return 6800.0, "fallback"


def kernel_source_hash():
    """Hash of the kernel sources' code (comments and layout ignored), which
    ties a committed ncu record to the kernels it was taken on."""
    h = hashlib.sha256()
    for f in ("jpsi_kernels.cu", "jpsi_device.cuh", "jpsi_internal.h"):
        src = open(os.path.join(ROOT, "paper_1810_11966_gb300", "csrc", f)).read()
        src = re.sub(r"/\*.*?\*/", " ", src, flags=re.S)
        src = re.sub(r"//[^\n]*", " ", src)
        h.update(" ".join(src.split()).encode())
    return h.hexdigest()[:16]


def ncu_record(kernel, workload, key):
    """A per-event figure (`key`) of `kernel` from the committed ncu summary,
    if it was taken on the current kernel source; else None."""
    p = os.path.join(ROOT, "profiles", "ncu_traffic.json")
    if not os.path.exists(p):
        return None
    d = json.load(open(p))
    e = d.get(kernel, {}).get(workload)
    if not e or e.get("source_hash") != kernel_source_hash() or key not in e:
        return None
    return float(e[key])


def ncu_traffic(kernel, workload):
    """DRAM bytes per event of `kernel` (ncu dram__bytes_read + write)."""
    return ncu_record(kernel, workload, "dram_bytes_per_event")


def issue_roofline(inst_per_event, n_events, kernel_ms, n_sm, sm_mhz):
    """Issue-slot roofline of a kernel: warp instructions per second against
    one instruction per cycle on each of the 4 schedulers of every SM at the
    SM clock seen under load."""
    peak = n_sm * 4 * sm_mhz * 1e6
    out = {"unit": "warp-inst/s", "peak": peak, "peak_kind": f"{n_sm} SMs x 4 schedulers x {sm_mhz:.0f} MHz",
           "inst_per_event": inst_per_event, "achieved": None, "frac": None}
    if inst_per_event is not None:
        out["achieved"] = inst_per_event * n_events / (kernel_ms / 1000.0)
        out["frac"] = out["achieved"] / peak
    return out


def algorithmic_bytes(n_events, n_hits, S, offsets=None, trigger=None):
    """Bytes the counting kernel must move at least: every processed hit read
    once (12 B), the CSR offsets that locate them (4 B each), per-unit counts
    (4 B), track count (4 B) and the per-event class byte.  CHAIN processes
    every station; PAPER (trigger given, with the host offsets) only the
    trigger station: its hits and its 4 offsets per event."""
    out = 4 * n_events * S + 4 * n_events + n_events
    if trigger is None:
        return 12 * n_hits + 4 * (n_events * 3 * S + 1) + out
    first = np.arange(n_events, dtype=np.int64) * 3 * S + 3 * trigger
    hits = int((offsets[first + 3].astype(np.int64) - offsets[first]).sum())
    return 12 * hits + 4 * 4 * n_events + out


def cpu_baseline(workload, params_kw, n_events, n_single=None, threads=None):
    """The oracle as it stands, on the host cores, over a bounded sample; and
    on one thread over the first n_single events of it."""
    import oracle
    import synth
    threads = threads or (os.cpu_count() or 1)
    b = synth.generate(workload, 0, n_events)
    p = oracle.params(**params_kw)
    t0 = time.perf_counter()
    r = oracle.run(p, b, triplets=True, n_threads=threads)
    dt = time.perf_counter() - t0
    assert r["status"] == 0
    out = {"value": n_events / dt, "unit": UNIT, "cores": threads, "kind": "oracle",
           "sample": f"events [0, {n_events}) of {workload}, counts + triplet lists, {threads} threads, "
                     f"{dt:.2f} s wall"}
    if n_single:
        b1 = synth.generate(workload, 0, n_single)
        t0 = time.perf_counter()
        r = oracle.run(p, b1, triplets=True, n_threads=1)
        dt1 = time.perf_counter() - t0
        assert r["status"] == 0
        out["single_thread"] = {"value": n_single / dt1, "unit": UNIT, "events": n_single, "wall_s": round(dt1, 3)}
    return out


def reference_arm(args, rank, world):
    """--impl reference: the oracle on the host cores, each step a bounded
    sample of the same workload; rank 0 only."""
    if rank != 0:
        return
    import oracle
    import synth
    w = synth.WORKLOADS[args.workload]
    if w.name == "poisson100_stream":
        return reference_arm_stream(args, w, world)
    threads = os.cpu_count() or 1
    n = args.ref_events
    b = synth.generate(w, 0, n)
    p = oracle.params(**params_kw(args, w))
    times = []
    for i in range(args.warmup + args.steps):
        t0 = time.perf_counter()
        r = oracle.run(p, b, triplets=True, n_threads=threads)
        dt = time.perf_counter() - t0
        assert r["status"] == 0
        if i >= args.warmup:
            times.append(dt)
    tot = sum(times)
    v = n * len(times) / tot
    line = {"impl": "reference", "metric": METRIC, "value": v, "unit": UNIT, "n_gpus": world, "steps": args.steps,
            "warmup": args.warmup, "ms_per_step": 1000 * tot / len(times), "higher_is_better": True,
            "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": w.name, "events_per_step": n, "stations": w.n_stations, "mode": args.mode},
            "cpu_baseline": {"value": v, "unit": UNIT, "cores": threads, "kind": "oracle",
                             "sample": f"events [0, {n}) of {w.name} per step"},
            "e2e": {"value": v, "unit": UNIT, "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def reference_arm_stream(args, w, world):
    """--impl reference on the free-streaming workload: the oracle's
    free-streaming selection over the first --cpu-windows windows of a
    2000-collision timeslice of the same recipe, per step."""
    import synth
    ts = synth.timeslice(w, 0, 2000)
    vals = []
    for i in range(args.warmup + args.steps):
        b = stream_cpu_baseline(ts, params_kw(args, w), n_windows=args.cpu_windows)
        if i >= args.warmup:
            vals.append(b["value"])
    v = sum(vals) / len(vals)
    line = {"impl": "reference", "metric": "collisions/s on 1 GB300, free-streaming timeslice (bit-exact accept bits)",
            "value": v, "unit": "collisions/s", "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": w.name, "windows_per_step": args.cpu_windows, "mode": args.mode},
            "cpu_baseline": {"value": v, "unit": "collisions/s", "cores": 1, "kind": "oracle",
                             "sample": b["sample"]},
            "e2e": {"value": v, "unit": "collisions/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0}}
    print(json.dumps(line), flush=True)


def percentiles(v, qs=(50, 99, 99.9)):
    a = np.sort(np.asarray(v, dtype=np.float64))
    return {f"p{q:g}": float(a[min(len(a) - 1, int(np.ceil(q / 100 * len(a))) - 1)]) for q in qs}


def canonical_rows(torch, trip_off, rows):
    """Triplet rows (n x 3) grouped by unit through the CSR `trip_off`, each
    unit's rows sorted lexicographically: equal for two outputs exactly when
    they hold the same rows per unit, whatever their order inside a unit."""
    rows = rows.to(torch.int64)
    n = rows.shape[0]
    unit = torch.repeat_interleave(torch.arange(trip_off.numel() - 1, device=trip_off.device),
                                   trip_off[1:] - trip_off[:-1])
    order = torch.arange(n, device=rows.device)
    for key in (rows[:, 2], rows[:, 1], rows[:, 0], unit):  # stable sorts, least significant key first
        order = order[torch.sort(key[order], stable=True)[1]]
    return rows[order]


def serve_slices_from_device(jp, torch, dev, p, slices, n_slots):
    """The same device-resident timeslices served through jpsi_serve_* with
    device batches and device outputs: while one slot waits on its host
    round trips or its kernels' tails, another slot's kernels run.  The slots
    read the timeslices and write the outputs in place.  One untimed pass (graph
    capture in every slot), then three timed passes of all timeslices, each
    from the first submit to the last completion (host wall clock, the device
    synchronised before); every served result is compared with the jpsi_run
    sweep's outputs (accept bits, track counts, offsets, and the triplet rows
    of each unit as a set: their order inside a unit is unspecified)."""
    torch.cuda.synchronize()

    def canon(s_):  # accept bits, counts, offsets, and the rows sorted inside each unit
        toff, n = s_[5], int(s_[2].trip_needed)
        return s_[3].clone(), s_[4].clone(), toff.clone(), canonical_rows(torch, toff, s_[6][:n])

    ref = [canon(s_) for s_ in slices]
    ctx = jp.Context(p, device=dev.index, hbm_budget=64 << 30)
    ev_max = max(int(s_[1].n_events) for s_ in slices)
    hits_max = max(int(s_[1].n_hits) for s_ in slices)
    cap = max(int(s_[2].trip_needed) for s_ in slices)
    ctx.check(jp.jpsi_serve_start(ctx.ctx, n_slots, ev_max, hits_max, cap))

    def one_pass():
        tickets, lat = [], []
        for s_ in slices:  # a submit blocks while every slot is busy
            s, tk = jp.jpsi_serve_submit(ctx.ctx, s_[1], s_[2])
            ctx.check(s)
            tickets.append(tk)
        for tk in tickets:
            ws, rs, lt = jp.jpsi_serve_wait(ctx.ctx, tk, 60000)
            ctx.check(ws)
            ctx.check(rs)
            lat.append(lt * 1000.0)
        return lat

    one_pass()
    torch.cuda.synchronize()
    ms, lat = [], []
    for _ in range(3):
        t0 = time.perf_counter()
        lat += one_pass()
        ms.append((time.perf_counter() - t0) * 1000.0)
    torch.cuda.synchronize()
    same = all(all(torch.equal(a, b) for a, b in zip(r, canon(s_))) for r, s_ in zip(ref, slices))
    ctx.check(jp.jpsi_serve_stop(ctx.ctx))
    ctx.close()
    n_ev = sum(int(s_[1].n_events) for s_ in slices)
    med = statistics.median(ms)
    return {"value": n_ev / (med / 1000.0), "unit": UNIT, "ms_total_median": med, "ms_total_passes": ms,
            "slots": n_slots, "slot_latency_ms": percentiles(lat, (50, 99)),
            "equal_to_jpsi_run": bool(same),
            "timing": "host wall clock per pass of every timeslice, first submit to last completion; "
                      "batches and outputs in device memory, used in place by the slots; median of 3 passes"}


def run_timeslices(args, w, dev, jp, torch):
    """Uneven timeslices (log-normal multiplicities): one jpsi_run per
    timeslice (persistent kernels replayed from the captured graph) against
    one jpsi_run_plain per timeslice, all data resident; beside them the same
    timeslices served from device memory over the serving slots."""
    import synth
    sizes = synth.timeslice_sizes(w, args.slices)
    starts = np.concatenate([[0], np.cumsum(sizes)[:-1]])
    p = jp.params(**params_kw(args, w))
    ctx = jp.Context(p, device=dev.index, hbm_budget=64 << 30)
    st = torch.cuda.current_stream(dev).cuda_stream
    slices = []
    t0 = time.perf_counter()
    n_hits_tot = 0
    for e0, n in zip(starts, sizes):
        b = synth.generate(w, int(e0), int(n))
        d = {k: torch.from_numpy(b[k]).to(dev) for k in ("x", "y", "z", "offsets")}
        batch = jp.make_batch(d["x"], d["y"], d["z"], d["offsets"], int(n), b["n_hits"])
        nu = int(n) * w.n_stations
        o = jp.jpsi_outputs()
        acc = torch.empty((int(n) + 31) // 32, dtype=torch.int32, device=dev)
        tc = torch.empty(int(n), dtype=torch.int32, device=dev)
        toff = torch.empty(nu + 1, dtype=torch.int64, device=dev)
        o.accept_bits, o.track_counts, o.trip_off = acc.data_ptr(), tc.data_ptr(), toff.data_ptr()
        ctx.check(jp.jpsi_run(ctx.ctx, batch, o, st))
        trip = torch.empty((max(o.trip_needed, 1), 3), dtype=torch.int32, device=dev)
        o.triplets, o.trip_capacity = trip.data_ptr(), o.trip_needed
        slices.append((d, batch, o, acc, tc, toff, trip))
        n_hits_tot += b["n_hits"]
    gen_s = time.perf_counter() - t0
    # the autotuner picks the batched form's launch shape on one timeslice
    mid = slices[len(slices) // 2]
    if not args.no_autotune:
        ctx.check(jp.jpsi_autotune(ctx.ctx, mid[1]))
    shape_t = jp.jpsi_timing_get(ctx.ctx)
    shape = {"warps_per_block": int(shape_t.light_wpb), "events_per_grab": int(shape_t.light_grab),
             "autotuned": not args.no_autotune}
    stream = torch.cuda.current_stream(dev)

    def sweep(fn):
        for s_ in slices:  # warm-up (graph capture, scratch growth)
            ctx.check(fn(ctx.ctx, s_[1], s_[2], st))
        torch.cuda.synchronize()
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(len(slices) + 1)]
        jp.jpsi_timing_enable(ctx.ctx, True)
        ev[0].record(stream)
        for i, s_ in enumerate(slices):
            ctx.check(fn(ctx.ctx, s_[1], s_[2], st))
            ev[i + 1].record(stream)
        torch.cuda.synchronize()
        tm = jp.jpsi_timing_get(ctx.ctx)
        jp.jpsi_timing_enable(ctx.ctx, False)
        per = [ev[i].elapsed_time(ev[i + 1]) for i in range(len(slices))]
        return sum(per), per, tm

    clocks = Clocks(dev.index)
    clocks.start()
    tb, per_b, tm_b = sweep(jp.jpsi_run)
    clk = clocks.stop()
    tp, per_p, _ = sweep(jp.jpsi_run_plain)
    ctx.close()
    clocks = Clocks(dev.index)
    clocks.start()
    slot_counts = [int(v) for v in args.served_slots.split(",")] if args.served_slots else [args.slots]
    by_slots = {n: serve_slices_from_device(jp, torch, dev, p, slices, n) for n in slot_counts}
    served = by_slots.get(args.slots, by_slots[slot_counts[0]])
    served["clocks"] = clocks.stop()
    n_ev = int(sizes.sum())
    # the counting phase of every timeslice (all tiles) against HBM: each hit
    # read once, offsets, unit and track counts, class bytes
    alg = algorithmic_bytes(n_ev, n_hits_tot, w.n_stations)
    count_ms = tm_b.light_ms + tm_b.count_rest_ms
    tpe = ncu_traffic("counting_phase", w.name)
    peak, peak_kind = measured_peaks()
    achieved = alg / (count_ms / 1000.0) / 1e9
    line = {"metric": METRIC, "value": n_ev / (tb / 1000), "unit": UNIT, "n_gpus": 1, "steps": 1, "warmup": 1,
            "ms_per_step": tb, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": w.name, "timeslices": len(sizes), "events": n_ev, "hits": n_hits_tot,
                       "slice_events_min": int(sizes.min()), "slice_events_max": int(sizes.max()),
                       "mode": args.mode, "window_cm": w.window, "launch_shape": shape},
            "plain": {"value": n_ev / (tp / 1000), "ms_total": tp},
            "speedup_batched_vs_plain": tp / tb,
            "slice_latency_ms": {"batched": percentiles(per_b, (50, 99)), "plain": percentiles(per_p, (50, 99))},
            "phases_ms": {"light_count": tm_b.light_ms, "count_rest": tm_b.count_rest_ms, "emit": tm_b.emit_ms},
            "roofline": {"bound": "hbm", "kernel": "counting phase (k_light, k_medium, k_sort_heavy, k_heavy, "
                         "k_heavy_units, k_heavy_final, k_generic, k_accept, scan)", "achieved": achieved,
                         "peak": peak, "peak_kind": peak_kind, "unit": "GB/s", "frac": achieved / peak,
                         "traffic": None if tpe is None else tpe * n_ev, "algorithmic_bytes": alg,
                         "per_event_figures": "ncu on the counting pass of timeslice 0, scaled by the events",
                         "issue": issue_roofline(ncu_record("counting_phase", w.name, "inst_per_event"), n_ev,
                                                 count_ms, torch.cuda.get_device_properties(dev).multi_processor_count,
                                                 clk.get("sm_mhz") or clk.get("sm_max_mhz") or 2070.0)},
            "served_from_device": served,
            "served_by_slots": {str(n): {k: r[k] for k in ("value", "ms_total_median", "slot_latency_ms",
                                                          "equal_to_jpsi_run")} for n, r in by_slots.items()},
            "gpu_launches": int(tm_b.kernel_launches), "clocks": clk, "generate_s": gen_s}
    if not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(w.name, params_kw(args, w), 20_000, n_single=2_000)
    print(json.dumps(line), flush=True)


def run_free_stream(args, w, dev, jp, torch):
    """A free-streaming timeslice (hits with times, no event association):
    jpsi_run_stream builds one event per time window on the device and runs
    the selection with the time tests; the metric is collisions per second.
    Device-resident steps, then end to end from pinned host buffers (the
    timeslice's copies in, the outputs' copies out, inside the timed
    region)."""
    import synth
    t0 = time.perf_counter()
    ts = synth.timeslice(w, 0, args.events or w.n_events)
    gen_s = time.perf_counter() - t0
    n_coll, n_hits, S = ts["n_collisions"], ts["n_hits"], w.n_stations
    K = len(ts["bounds"]) - 1
    host = {k: torch.from_numpy(np.ascontiguousarray(ts[k])).pin_memory()
            for k in ("x", "y", "z", "t", "offsets", "bounds")}
    d = {k: v.to(dev) for k, v in host.items()}
    torch.cuda.synchronize()
    p = jp.params(**params_kw(args, w))
    ctx = jp.Context(p, device=dev.index, hbm_budget=64 << 30)
    stream = torch.cuda.current_stream(dev)
    st = stream.cuda_stream
    tsd = jp.make_timeslice(d["x"], d["y"], d["z"], d["t"], d["offsets"], d["bounds"], ts["dt"])
    nu = K * S
    acc = torch.empty((K + 31) // 32, dtype=torch.int32, device=dev)
    tc = torch.empty(K, dtype=torch.int32, device=dev)
    toff = torch.empty(nu + 1, dtype=torch.int64, device=dev)
    o = jp.jpsi_outputs()
    o.accept_bits, o.track_counts, o.trip_off = acc.data_ptr(), tc.data_ptr(), toff.data_ptr()
    ctx.check(jp.jpsi_run_stream(ctx.ctx, tsd, o, st))
    cap = o.trip_needed
    trip = torch.empty((max(cap, 1), 3), dtype=torch.int32, device=dev)
    o.triplets, o.trip_capacity = trip.data_ptr(), cap

    def timed(fn, steps, warmup):
        for _ in range(warmup):
            ctx.check(fn(ctx.ctx, tsd, o, st))
        torch.cuda.synchronize()
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(steps + 1)]
        jp.jpsi_timing_enable(ctx.ctx, True)
        ev[0].record(stream)
        for i in range(steps):
            ctx.check(fn(ctx.ctx, tsd, o, st))
            ev[i + 1].record(stream)
        torch.cuda.synchronize()
        tm = jp.jpsi_timing_get(ctx.ctx)
        jp.jpsi_timing_enable(ctx.ctx, False)
        return ev[0].elapsed_time(ev[steps]), [ev[i].elapsed_time(ev[i + 1]) for i in range(steps)], tm

    clocks = Clocks(dev.index)
    clocks.start()
    tot_b, per_b, tm_b = timed(jp.jpsi_run_stream, args.steps, args.warmup)
    clk = clocks.stop()
    tot_p, per_p, _ = timed(jp.jpsi_run_stream_plain, max(args.steps // 2, 3), 3)
    ref_tc = tc.cpu().numpy().copy()

    # end to end: the timeslice from pinned host memory, the outputs back
    hout = {"acc": torch.empty_like(acc, device="cpu").pin_memory(),
            "tc": torch.empty_like(tc, device="cpu").pin_memory(),
            "toff": torch.empty_like(toff, device="cpu").pin_memory(),
            "trip": torch.empty_like(trip, device="cpu").pin_memory()}

    def e2e_step():
        for k in ("x", "y", "z", "t", "offsets", "bounds"):
            d[k].copy_(host[k], non_blocking=True)
        ctx.check(jp.jpsi_run_stream(ctx.ctx, tsd, o, st))
        hout["acc"].copy_(acc, non_blocking=True)
        hout["tc"].copy_(tc, non_blocking=True)
        hout["toff"].copy_(toff, non_blocking=True)
        hout["trip"][:cap].copy_(trip[:cap], non_blocking=True)
        stream.synchronize()

    for _ in range(3):
        e2e_step()
    e2e_t = []
    for _ in range(args.e2e_steps):
        t1 = time.perf_counter()
        e2e_step()
        e2e_t.append(time.perf_counter() - t1)
    assert np.array_equal(hout["tc"].numpy(), ref_tc)
    e2e_mean = sum(e2e_t) / len(e2e_t)
    h2d = 16 * n_hits + 4 * (3 * S + 1) + 4 * (K + 1)
    d2h = 4 * ((K + 31) // 32) + 4 * K + 8 * (nu + 1) + 12 * cap

    ms_b = tot_b / args.steps
    ms_p = tot_p / len(per_p)
    runs = max(tm_b.runs, 1)
    win_ms = tm_b.window_ms / runs
    # the event-building phase moves at least: t and z of every hit (checks; the
    # hits themselves stay where they are), the ranges (first hit, size, offset in
    # 64 and 32 bits, shift), and each triplet row read and written once by the
    # mapping back
    built = jp_window_hits(ts, p)
    alg = 8 * n_hits + K * 3 * S * (4 + 4 + 8 + 4 + 4) + 24 * cap
    peak, peak_kind = measured_peaks()
    achieved = alg / (win_ms / 1000.0) / 1e9
    per_sorted = sorted(per_b)
    line = {
        "metric": "collisions/s on 1 GB300, free-streaming timeslice (bit-exact accept bits)",
        "value": n_coll / (ms_b / 1000.0), "unit": "collisions/s", "n_gpus": 1, "steps": args.steps,
        "warmup": args.warmup, "ms_per_step": ms_b, "higher_is_better": True, "scaling": "weak",
        "vs_baseline": None, "dtype": "f32", "data": "synthetic",
        "config": {"workload": w.name, "collisions": n_coll, "hits": n_hits, "windows": K,
                   "window_ns": float(ts["bounds"][1] - ts["bounds"][0]), "dt_ns": ts["dt"],
                   "rate_hz": w.extra["rate_hz"], "sigma_t_ns": w.extra["sigma_t_ns"], "mode": args.mode,
                   "window_batch_hits": built, "form": "batched (persistent kernels + CUDA graph)",
                   "l2": f"inputs ({16 * n_hits / 1e9:.1f} GB) larger than L2; no flush"},
        "windows_per_s": K / (ms_b / 1000.0), "hits_per_s": n_hits / (ms_b / 1000.0),
        "plain": {"value": n_coll / (ms_p / 1000.0), "ms_per_step": ms_p},
        "latency_ms": {"p50": per_sorted[len(per_sorted) // 2], "max": per_sorted[-1]},
        "phases_ms": {"event_building": win_ms, "light_count": tm_b.light_ms / runs,
                      "count_rest": tm_b.count_rest_ms / runs, "emit": tm_b.emit_ms / runs},
        "roofline": {"bound": "hbm", "kernel": "event building (k_win_check, k_win_ranges, scan, k_win_place, "
                     "k_win_rows)", "achieved": achieved, "peak": peak, "peak_kind": peak_kind, "unit": "GB/s",
                     "frac": achieved / peak, "traffic": None, "algorithmic_bytes": alg},
        "e2e": {"value": n_coll / e2e_mean, "unit": "collisions/s", "h2d_bytes_per_step": h2d,
                "d2h_bytes_per_step": d2h, "ms_per_step": 1000 * e2e_mean,
                "ms_samples": [round(1000 * v, 2) for v in e2e_t]},
        "gpu_launches": int(tm_b.kernel_launches), "clocks": clk, "triplets_per_step": cap,
        "accepted_windows": int(np.count_nonzero(ref_tc >= p.min_candidates)), "generate_s": gen_s,
    }
    if not args.no_cpu_baseline:
        line["cpu_baseline"] = stream_cpu_baseline(ts, params_kw(args, w), n_windows=args.cpu_windows)
    print(json.dumps(line), flush=True)
    ctx.close()


def jp_window_hits(ts, p):
    """Hits of the window batch (the ranges the library selects from), counted on
    the host from the timeslice: the trigger station's [b_k, fl32(b_k+1 + dt)],
    the other stations (CHAIN) from just below b_k - dt to the same end."""
    t, off, b = ts["t"], ts["offsets"], ts["bounds"].astype(np.float32)
    dt = np.float32(ts["dt"])
    end = (b[1:] + dt).astype(np.float32)
    total = 0
    for g in range(len(off) - 1):
        s = g // 3
        if p.mode == 0 and s != p.trigger_station:
            continue
        tg = t[off[g]:off[g + 1]]
        b64 = b[:-1].astype(np.float64)
        lod = (b64 - float(dt)) - (1e-6 * (np.abs(b64) + float(dt)) + 1e-30)
        lo = b[:-1] if s == p.trigger_station else np.nextafter(lod.astype(np.float32), np.float32(-np.inf))
        total += int((np.searchsorted(tg, end, side="right") - np.searchsorted(tg, lo, side="left")).clip(0).sum())
    return total


def stream_cpu_baseline(ts, kw, n_windows=12):
    """The oracle's free-streaming selection, as it stands, on a bounded
    sample: the first n_windows windows of the timeslice (one host thread),
    scaled to collisions/s by the collisions whose time lies in them."""
    import oracle
    p = oracle.params(kw["n_stations"], kw["mode"], t_xz=kw["t_xz"], t_yz=kw["t_yz"])
    b = ts["bounds"][: n_windows + 1]
    t0 = time.perf_counter()
    r = oracle.stream(p, ts, b, ts["dt"])
    sec = time.perf_counter() - t0
    assert r["status"] == 0
    ct = ts["collision_times"]
    n = int(np.count_nonzero((ct >= b[0]) & (ct < b[-1])))
    return {"value": n / sec, "unit": "collisions/s", "cores": 1, "kind": "oracle",
            "sample": f"windows 0..{n_windows - 1} ({n} collisions) of the timeslice, counts and rows, "
                      f"{sec:.1f} s on one core"}


def run_serving(args, w, dev, jp, torch):
    """Continuous batching: timeslices of U[2e3, 2e5] events arrive as a
    Poisson process; jpsi_serve_submit admits each into a resident device slot
    as soon as one frees up (a blocking submit is the back-pressure) and runs
    it on that slot's stream while other slots copy or compute.  Latency =
    completion (outputs in host memory) - arrival.  Offered loads: the
    workload's 10^7 events/s, saturation (all requests at t=0), and 50/80/95 %
    of the saturated throughput; each load is `--requests` requests long.
    Requests cycle over a pool of distinct timeslices and over a ring of
    output buffers (a buffer is reused once its earlier request was waited
    for); every served result is compared with the same timeslice run alone
    (accept bits exactly, track counts and triplet total)."""
    import threading

    import synth
    n_req = args.requests
    pool_n = min(args.pool, n_req)
    sizes_all = synth.timeslice_sizes(w, pool_n)
    p = jp.params(**params_kw(args, w))
    ctx = jp.Context(p, device=dev.index, hbm_budget=args.serve_budget_gb << 30)
    st = torch.cuda.current_stream(dev).cuda_stream
    S = w.n_stations
    pool, e0 = [], 0
    t0 = time.perf_counter()
    for i in range(pool_n):
        n = int(sizes_all[i])
        b = synth.generate(w, e0, n)
        e0 += n
        h = {k: torch.from_numpy(b[k]).pin_memory() for k in ("x", "y", "z", "offsets")}
        # the timeslice alone: exact triplet count (slot sizing) and the
        # reference result of the isolation check
        d = {k: v.to(dev) for k, v in h.items()}
        r = ctx.select(d["x"], d["y"], d["z"], d["offsets"], n)
        ctx.check(r["status"])
        pool.append({"h": h, "n": n, "hits": b["n_hits"], "trip": r["trip_needed"],
                     "acc": r["accept_bits"].cpu().numpy().copy(), "tc_sum": int(r["track_counts"].sum().item())})
        del d, r
    gen_s = time.perf_counter() - t0
    torch.cuda.empty_cache()
    slot_events = max(q["n"] for q in pool)
    slot_hits = max(q["hits"] for q in pool)
    slot_trip = max(q["trip"] for q in pool)
    ctx.check(jp.jpsi_serve_start(ctx.ctx, args.slots, slot_events, slot_hits, slot_trip))
    # enough output buffers that buffer reuse never holds a submission back
    # behind a slow earlier request (a short ring coupled the requests)
    ring_n = max(64, 4 * args.slots)
    ring = []
    for _ in range(ring_n):
        ob = {"acc": torch.empty((slot_events + 31) // 32, dtype=torch.int32, pin_memory=True),
              "tc": torch.empty(slot_events, dtype=torch.int32, pin_memory=True),
              "toff": torch.empty(slot_events * S + 1, dtype=torch.int64, pin_memory=True),
              "trip": torch.empty((max(slot_trip, 1), 3), dtype=torch.int32, pin_memory=True)}
        ring.append(ob)
    batches = [jp.make_batch(q["h"]["x"], q["h"]["y"], q["h"]["z"], q["h"]["offsets"], q["n"], q["hits"])
               for q in pool]
    n_events = sum(pool[i % pool_n]["n"] for i in range(n_req))

    def outputs(i):
        q, ob = pool[i % pool_n], ring[i % ring_n]
        o = jp.jpsi_outputs()
        o.accept_bits, o.track_counts = ob["acc"].data_ptr(), ob["tc"].data_ptr()
        o.trip_off, o.triplets, o.trip_capacity = ob["toff"].data_ptr(), ob["trip"].data_ptr(), q["trip"]
        return o

    def run_load(rate, check):
        mean = n_events / n_req
        if rate is None:
            arr = np.zeros(n_req)
        else:
            rng = np.random.Generator(np.random.PCG64(w.seed * 7919 + int(rate)))
            arr = np.cumsum(rng.exponential(mean / rate, size=n_req))
            arr -= arr[0]
        subs = [None] * n_req
        outs = [None] * n_req
        waited = [0]
        cv = threading.Condition()
        t_start = time.perf_counter() + 0.05

        def submitter():
            for i in range(n_req):
                with cv:  # the ring buffer of request i is free once request i - ring_n was waited for
                    cv.wait_for(lambda: waited[0] > i - ring_n)
                delay = t_start + arr[i] - time.perf_counter()
                if delay > 0:
                    time.sleep(delay)
                tc0 = time.perf_counter()
                outs[i] = outputs(i)
                s_, tk = jp.jpsi_serve_submit(ctx.ctx, batches[i % pool_n], outs[i])
                subs[i] = (s_, tk, tc0 - (t_start + arr[i]))
        th = threading.Thread(target=submitter)
        th.start()
        lat, done, mismatches = [], [], 0
        for i in range(n_req):
            while subs[i] is None:
                time.sleep(0.0002)
            s_, tk, queued = subs[i]
            assert s_ == 0, s_
            ws, rs, lat_lib = jp.jpsi_serve_wait(ctx.ctx, tk, 60000)
            assert ws == 0 and rs == 0, (ws, rs)
            lat.append(queued + lat_lib)
            done.append(arr[i] + queued + lat_lib)
            if check:
                q, ob = pool[i % pool_n], ring[i % ring_n]
                nw = (q["n"] + 31) // 32
                same = (np.array_equal(ob["acc"].numpy()[:nw], q["acc"]) and
                        int(ob["tc"][: q["n"]].sum().item()) == q["tc_sum"] and
                        outs[i].trip_needed == q["trip"])
                mismatches += 0 if same else 1
            with cv:
                waited[0] = i + 1
                cv.notify_all()
        th.join()
        span = max(done)
        out = {"offered_events_per_s": None if rate is None else rate, "sustained_events_per_s": n_events / span,
               "requests": n_req, "latency_ms": {k: 1000 * v for k, v in percentiles(lat).items()}}
        if check:
            out["results_equal_solo"] = mismatches == 0
        return out

    run_load(None, False)  # warm-up: graphs, buffers
    jp.jpsi_timing_enable(ctx.ctx, True)
    sat = run_load(None, True)
    tm = jp.jpsi_timing_get(ctx.ctx)
    cap = sat["sustained_events_per_s"]
    loads = [run_load(w.extra["rate_events_per_s"], True)]
    for f in (0.5, 0.8, 0.95):
        r = run_load(f * cap, True)
        r["fraction_of_saturation"] = f
        loads.append(r)
    ctx.check(jp.jpsi_serve_stop(ctx.ctx))
    line = {"metric": METRIC, "value": cap, "unit": UNIT, "n_gpus": 1, "steps": len(loads) + 2, "warmup": 1,
            "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32", "data": "synthetic",
            "config": {"workload": w.name, "requests_per_load": n_req, "distinct_timeslices": pool_n,
                       "events_per_load": n_events, "slots": args.slots, "slot_events": slot_events,
                       "slot_hits": slot_hits, "hbm_budget_gb": args.serve_budget_gb, "mode": args.mode},
            "saturation": sat, "loads": loads,
            "kernel_launches_per_request": tm.kernel_launches / max(tm.runs, 1),
            "isolation": all(r.get("results_equal_solo", True) for r in [sat] + loads),
            "generate_s": gen_s}
    if not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(w.name, params_kw(args, w), 20_000, n_single=2_000)
    print(json.dumps(line), flush=True)
    ctx.close()


def run_stress(args, w, dev, jp, torch):
    """Combinatorial stress workload (6 stations, Poisson(1500) per layer,
    window 1.0 cm): batches of at most 75 000 events (int32 CSR offsets), each
    run once to size its triplet buffer and then timed; the triplet lists are
    written in full."""
    import synth
    n_total = args.events or w.n_events
    chunk = min(args.chunk, 75_000)
    p = jp.params(**params_kw(args, w))
    ctx = jp.Context(p, device=dev.index, hbm_budget=args.stress_budget_gb << 30)
    st = torch.cuda.current_stream(dev).cuda_stream
    stream = torch.cuda.current_stream(dev)
    tot_ms, trips, hits, gen_s = 0.0, 0, 0, 0.0
    for e0 in range(0, n_total, chunk):
        n = min(chunk, n_total - e0)
        t0 = time.perf_counter()
        b = synth.generate(w, e0, n)
        gen_s += time.perf_counter() - t0
        d = {k: torch.from_numpy(b[k]).to(dev) for k in ("x", "y", "z", "offsets")}
        hits += b["n_hits"]
        del b
        batch = jp.make_batch(d["x"], d["y"], d["z"], d["offsets"], n, int(d["x"].numel()))
        o = jp.jpsi_outputs()
        acc = torch.empty((n + 31) // 32, dtype=torch.int32, device=dev)
        tc = torch.empty(n, dtype=torch.int32, device=dev)
        toff = torch.empty(n * w.n_stations + 1, dtype=torch.int64, device=dev)
        o.accept_bits, o.track_counts, o.trip_off = acc.data_ptr(), tc.data_ptr(), toff.data_ptr()
        ctx.check(jp.jpsi_run(ctx.ctx, batch, o, st))
        trip = torch.empty((max(o.trip_needed, 1), 3), dtype=torch.int32, device=dev)
        o.triplets, o.trip_capacity = trip.data_ptr(), o.trip_needed
        ctx.check(jp.jpsi_run(ctx.ctx, batch, o, st))  # warm: sizes the triplet record
        e_a, e_b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        torch.cuda.synchronize()
        e_a.record(stream)
        ctx.check(jp.jpsi_run(ctx.ctx, batch, o, st))
        e_b.record(stream)
        torch.cuda.synchronize()
        tot_ms += e_a.elapsed_time(e_b)
        trips += o.trip_needed
        del d, trip, acc, tc, toff
        torch.cuda.empty_cache()
    line = {"metric": METRIC, "value": n_total / (tot_ms / 1000), "unit": UNIT, "n_gpus": 1, "steps": 1, "warmup": 1,
            "ms_per_step": tot_ms, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
            "data": "synthetic",
            "config": {"workload": w.name, "events": n_total, "chunk_events": chunk, "hits": hits,
                       "stations": w.n_stations, "window_cm": w.window, "mode": args.mode},
            "triplets": trips, "triplets_per_s": trips / (tot_ms / 1000), "generate_s": gen_s}
    if not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(w.name, params_kw(args, w), 32, n_single=4)
    print(json.dumps(line), flush=True)
    ctx.close()


def signal_diagnostic(w, e0, n, acc_words):
    """Synthetic signal-finding rate, a diagnostic (the paper's efficiency
    study needs its simulation samples): the fraction of events accepted
    among those generated with two, one and no muons, over events [e0, e0+n)
    of the workload, from the accept bits of the run."""
    import synth
    b = synth.generate(w, e0, n, truth=True)
    counts = np.diff(b["offsets"].astype(np.int64)).reshape(n, -1).sum(axis=1)
    ev = np.repeat(np.arange(n), counts)
    n_mu = np.zeros(n, np.int64)
    np.maximum.at(n_mu, ev, b["truth"].astype(np.int64))  # muons are numbered 1, 2 within an event
    bits = (acc_words.view(np.uint32)[np.arange(n) // 32] >> (np.arange(n) % 32).astype(np.uint32)) & 1
    out = {"events": n}
    for k in (2, 1, 0):
        sel = n_mu == k
        out[f"events_{k}mu"] = int(sel.sum())
        out[f"accepted_{k}mu"] = float(bits[sel].mean()) if sel.any() else None
    return out


def params_kw(args, w):
    t = w.window ** 2
    return {"n_stations": w.n_stations, "mode": 1 if args.mode == "chain" else 0, "t_xz": t, "t_yz": t}


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=40)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="poisson100_1m")
    ap.add_argument("--events", type=int, default=None, help="events per rank (default: the workload's)")
    ap.add_argument("--mode", default="chain", choices=["chain", "paper"])
    ap.add_argument("--e2e-steps", type=int, default=8)
    ap.add_argument("--cpu-events", type=int, default=100_000)
    ap.add_argument("--ref-events", type=int, default=40_000)
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--profile-steps", type=int, default=0, help="(for ncu) run this many steps and exit")
    ap.add_argument("--slices", type=int, default=None, help="timeslices (timeslice/stream workloads)")
    ap.add_argument("--no-autotune", action="store_true")
    ap.add_argument("--chunk", type=int, default=50_000, help="events per batch (stress workload)")
    ap.add_argument("--stress-budget-gb", type=int, default=160)
    ap.add_argument("--pool", type=int, default=8, help="distinct timeslices generated for the stream workload")
    ap.add_argument("--slots", type=int, default=5)
    ap.add_argument("--served-slots", default=None,
                    help="timeslice workload: comma-separated slot counts to serve from device memory (default: --slots)")
    ap.add_argument("--requests", type=int, default=1000, help="requests per offered load (stream workload)")
    ap.add_argument("--serve-budget-gb", type=int, default=16)
    ap.add_argument("--cpu-windows", type=int, default=12, help="windows of the stream workload's CPU sample")
    args = ap.parse_args()
    rank, world, local = dist_info()
    if args.warmup < 3 and not args.profile_steps:
        raise SystemExit("--warmup must be >= 3")
    if args.impl == "reference":
        return reference_arm(args, rank, world)

    import torch

    import paper_1810_11966_gb300 as jp
    import synth

    torch.cuda.set_device(local)
    dev = torch.device("cuda", local)
    pg = None
    if world > 1:
        import torch.distributed as dist
        dist.init_process_group("gloo")
        pg = dist
    jp.load(build_if_missing=True)
    w = synth.WORKLOADS[args.workload]
    if w.name == "lognormal_timeslices":
        return run_timeslices(args, w, dev, jp, torch)
    if w.name == "lognormal_stream":
        return run_serving(args, w, dev, jp, torch)
    if w.name == "poisson1500_6st":
        return run_stress(args, w, dev, jp, torch)
    if w.name == "poisson100_stream":
        return run_free_stream(args, w, dev, jp, torch)
    n_ev = args.events or w.n_events
    S = w.n_stations

    # host batch in pinned memory (for the end-to-end leg), then resident copies
    t0 = time.perf_counter()
    e_first, _ = shard(rank, n_ev)
    counts = synth.layer_counts(w, e_first, n_ev)
    n_hits = int(counts.sum())
    pin = {k: torch.empty(n_hits, dtype=torch.float32, pin_memory=True) for k in ("x", "y", "z")}
    host = synth.generate(w, e_first, n_ev, out={k: v.numpy() for k, v in pin.items()})
    off_pin = torch.from_numpy(host["offsets"]).pin_memory()
    gen_s = time.perf_counter() - t0
    d = {k: pin[k].to(dev) for k in ("x", "y", "z")}
    d["offsets"] = off_pin.to(dev)
    torch.cuda.synchronize()

    p = jp.params(**params_kw(args, w))
    ctx = jp.Context(p, device=local, hbm_budget=64 << 30)
    stream = torch.cuda.current_stream(dev)
    st = stream.cuda_stream
    batch = jp.make_batch(d["x"], d["y"], d["z"], d["offsets"], n_ev, n_hits)

    # outputs, sized by a counting run
    nu = n_ev * S
    acc = torch.empty((n_ev + 31) // 32, dtype=torch.int32, device=dev)
    tc = torch.empty(n_ev, dtype=torch.int32, device=dev)
    toff = torch.empty(nu + 1, dtype=torch.int64, device=dev)
    o = jp.jpsi_outputs()
    o.accept_bits, o.track_counts, o.trip_off = acc.data_ptr(), tc.data_ptr(), toff.data_ptr()
    ctx.check(jp.jpsi_run(ctx.ctx, batch, o, st))
    cap = o.trip_needed
    trip = torch.empty((max(cap, 1), 3), dtype=torch.int32, device=dev)
    o.triplets, o.trip_capacity = trip.data_ptr(), cap

    if args.profile_steps:  # for ncu: the default launch shape, no autotuning launches
        for _ in range(args.profile_steps):
            ctx.check(jp.jpsi_run(ctx.ctx, batch, o, st))
        torch.cuda.synchronize()
        return

    # the autotuner picks the batched form's launch shape on this batch
    if not args.no_autotune:
        ctx.check(jp.jpsi_autotune(ctx.ctx, batch))
    shape_t = jp.jpsi_timing_get(ctx.ctx)
    shape = {"warps_per_block": int(shape_t.light_wpb), "events_per_grab": int(shape_t.light_grab),
             "autotuned": not args.no_autotune}

    def timed(run_fn, steps, warmup):
        for _ in range(warmup):
            ctx.check(run_fn(ctx.ctx, batch, o, st))
        torch.cuda.synchronize()
        if pg:
            pg.barrier()
        evs = [torch.cuda.Event(enable_timing=True) for _ in range(steps + 1)]
        jp.jpsi_timing_enable(ctx.ctx, True)
        evs[0].record(stream)
        for i in range(steps):
            ctx.check(run_fn(ctx.ctx, batch, o, st))
            evs[i + 1].record(stream)
        torch.cuda.synchronize()
        tm = jp.jpsi_timing_get(ctx.ctx)
        jp.jpsi_timing_enable(ctx.ctx, False)
        per = [evs[i].elapsed_time(evs[i + 1]) for i in range(steps)]
        tot = evs[0].elapsed_time(evs[steps])
        if pg:
            tot = max_over_ranks(tot, pg)
        return tot, per, tm

    clocks = Clocks(local)
    clocks.start()
    tot_b, per_b, tm_b = timed(jp.jpsi_run, args.steps, args.warmup)
    clk = clocks.stop()
    tot_p, per_p, tm_p = timed(jp.jpsi_run_plain, max(args.steps // 2, 3), 3)

    # end to end through the public API from pinned host buffers
    hb = jp.make_batch(pin["x"], pin["y"], pin["z"], off_pin, n_ev, n_hits)
    h_acc = torch.empty((n_ev + 31) // 32, dtype=torch.int32, pin_memory=True)
    h_tc = torch.empty(n_ev, dtype=torch.int32, pin_memory=True)
    h_to = torch.empty(nu + 1, dtype=torch.int64, pin_memory=True)
    h_tr = torch.empty((max(cap, 1), 3), dtype=torch.int32, pin_memory=True)
    ho = jp.jpsi_outputs()
    ho.accept_bits, ho.track_counts, ho.trip_off, ho.triplets = (h_acc.data_ptr(), h_tc.data_ptr(), h_to.data_ptr(),
                                                                 h_tr.data_ptr())
    ho.trip_capacity = cap
    for _ in range(3):
        ctx.check(jp.jpsi_run_host(ctx.ctx, hb, ho, st))
    e2e_t = []
    for _ in range(args.e2e_steps):
        t0 = time.perf_counter()
        ctx.check(jp.jpsi_run_host(ctx.ctx, hb, ho, st))
        e2e_t.append(time.perf_counter() - t0)
    e2e_mean = sum(e2e_t) / len(e2e_t)
    # the same from a per-layer geometry table (z = NULL; the generator puts
    # every hit on its layer's plane): 8 bytes per hit cross the host link
    table = np.array([np.float32(zs + (l - 1) * w.layer_dz) for zs in w.station_z for l in range(3)], np.float32)
    hbz = jp.make_batch(pin["x"], pin["y"], None, off_pin, n_ev, n_hits, z_layer=table)
    h_tc2 = h_tc.clone()
    for _ in range(3):
        ctx.check(jp.jpsi_run_host(ctx.ctx, hbz, ho, st))
    ez_t = []
    for _ in range(args.e2e_steps):
        t0 = time.perf_counter()
        ctx.check(jp.jpsi_run_host(ctx.ctx, hbz, ho, st))
        ez_t.append(time.perf_counter() - t0)
    assert np.array_equal(h_tc.numpy(), h_tc2.numpy())
    ez_mean = sum(ez_t) / len(ez_t)
    if pg:  # the job's end-to-end time is the slowest rank's
        e2e_mean = max_over_ranks(e2e_mean, pg)
        ez_mean = max_over_ranks(ez_mean, pg)
    h2d = 12 * n_hits + 4 * (n_ev * 3 * S + 1)
    d2h = 4 * ((n_ev + 31) // 32) + 4 * n_ev + 8 * (nu + 1) + 12 * cap
    assert np.array_equal(h_tc.numpy(), tc.cpu().numpy())

    ms_b = tot_b / args.steps
    ms_p = tot_p / len(per_p)
    value = world * n_ev / (ms_b / 1000.0)
    light_ms = tm_b.light_ms / max(tm_b.runs, 1)
    alg = (algorithmic_bytes(n_ev, n_hits, S) if args.mode == "chain" else
           algorithmic_bytes(n_ev, n_hits, S, offsets=host["offsets"], trigger=p.trigger_station))
    peak, peak_kind = measured_peaks()
    achieved = alg / (light_ms / 1000.0) / 1e9
    tpe = ncu_traffic("k_light_count", w.name)
    per_sorted = sorted(per_b)

    line = {
        "metric": METRIC, "value": value, "unit": UNIT, "n_gpus": world, "steps": args.steps, "warmup": args.warmup,
        "ms_per_step": ms_b, "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f32",
        "data": "synthetic",
        "config": {"workload": w.name, "n_events": n_ev, "stations": S, "mean_hits_per_event": n_hits / n_ev,
                   "mode": args.mode, "window_cm": w.window, "form": "batched (persistent kernels + CUDA graph)",
                   "l2": f"inputs ({12 * n_hits / 1e9:.1f} GB) larger than L2; no flush", "seed": w.seed,
                   "launch_shape": shape},
        "hits_per_s": world * n_hits / (ms_b / 1000.0),
        "median_step": {"events_per_s": world * n_ev / (per_sorted[len(per_sorted) // 2] / 1000.0),
                        "hits_per_s": world * n_hits / (per_sorted[len(per_sorted) // 2] / 1000.0)},
        "plain": {"value": world * n_ev / (ms_p / 1000.0), "ms_per_step": ms_p},
        "latency_ms": {"p50": per_sorted[len(per_sorted) // 2],
                       "p99": per_sorted[min(len(per_sorted) - 1, int(0.99 * len(per_sorted)))]},
        "phases_ms": {"light_count": light_ms, "count_rest": tm_b.count_rest_ms / max(tm_b.runs, 1),
                      "emit": tm_b.emit_ms / max(tm_b.runs, 1)},
        "roofline": {"bound": "hbm", "kernel": "k_light_count", "achieved": achieved, "peak": peak,
                     "peak_kind": peak_kind, "unit": "GB/s", "frac": achieved / peak,
                     "traffic": None if tpe is None else tpe * n_ev,
                     "algorithmic_bytes": alg,
                     "issue": issue_roofline(ncu_record("k_light_count", w.name, "inst_per_event"), n_ev, light_ms,
                                             torch.cuda.get_device_properties(dev).multi_processor_count,
                                             clk.get("sm_mhz") or clk.get("sm_max_mhz") or 2070.0)},
        "e2e": {"value": world * n_ev / e2e_mean, "unit": UNIT, "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h,
                "ms_per_step": 1000 * e2e_mean, "steps": len(e2e_t),
                "ms_median": 1000 * sorted(e2e_t)[len(e2e_t) // 2], "ms_min": 1000 * min(e2e_t),
                "ms_max": 1000 * max(e2e_t), "ms_samples": [round(1000 * v, 2) for v in e2e_t]},
        "e2e_layer_z": {"value": world * n_ev / ez_mean, "unit": UNIT,
                        "h2d_bytes_per_step": 8 * n_hits + 4 * (n_ev * 3 * S + 1) + 4 * 3 * S,
                        "d2h_bytes_per_step": d2h, "ms_per_step": 1000 * ez_mean,
                        "ms_samples": [round(1000 * v, 2) for v in ez_t],
                        "input": "x, y per hit + z per layer (jpsi_batch.z_layer); same results"},
        "gpu_launches": int(tm_b.kernel_launches),
        "clocks": clk,
        "triplets_per_step": cap,
        "generate_s": gen_s,
    }
    if rank == 0:
        line["signal_diagnostic"] = signal_diagnostic(w, e_first, min(100_000, n_ev), acc.cpu().numpy())
    if rank == 0 and not args.no_cpu_baseline:
        line["cpu_baseline"] = cpu_baseline(w.name, params_kw(args, w), min(args.cpu_events, n_ev),
                                            n_single=min(10_000, n_ev))
    if rank == 0:
        print(json.dumps(line), flush=True)
    ctx.close()
    if pg:
        pg.destroy_process_group()


if __name__ == "__main__":
    main()
