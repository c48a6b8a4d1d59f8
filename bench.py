#!/usr/bin/env python
"""Benchmark of the pLogP tuner on N GPUs of one node (one process per GPU).

A step is one pass of the whole path — plogp_select_best over the workload: table staging, g()
interpolation, all enabled Table 1 / Table 2 models, the segment-size search, the Scatter sums,
strategy selection and the decision-table stores.  The default workload is the batched
multi-network configuration (4096 seeded tables x P = 2..512 x 128 m x 32 s, all 13 strategies);
`--workload cfg3` times the exhaustive segment sweep instead.  With N > 1 every rank evaluates
its own 4096 tables (different seeds): weak scaling, no data-path collective.

The JSON line (ONE line, rank 0) carries the headline workload at top level and, at N = 1, a
`workloads` list with the other configurations timed in the same run (the exhaustive sweep, the
prediction call on the batched workload, and the three microsecond-scale configurations, marked
launch-bound), each with its own ms_per_step, cells/s and dominant-kernel roofline object.
`--impl reference` times the CPU oracle on a bounded sample of the same workload instead (rank 0
only).  Run plainly with `--gpus N` (no launcher) it starts the N ranks itself.
"""
from __future__ import annotations

import argparse
import json
import os
import statistics
import sys
import threading
import time

import numpy as np

ROOT = os.path.dirname(os.path.abspath(__file__))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

from paper_cs_0408034_b200 import workloads as wl  # noqa: E402

NOMINAL_FP64_FMA_RATE = 148 * 64 * 1.965e9  # SMs x FP64 lanes per SM x max SM clock
# dram__bytes_read.sum and dram__bytes_write.sum per launch from the ncu captures summarised under profiles/ (batched workload
# cut to 1024 tables).  Of the 0.87 GB that a kernel writes there, some 60 MB are still in the L2 when it ends, on any number of
# tables: a larger launch writes 13 B per cell and reads its tables more.  None while a kernel has changed since its last capture.
NCU_TRAFFIC_TABLES = 1024
NCU_TRAFFIC = {"decide_kernel": (1456896, 811407872), "scatter_kernel": (1700000, 812060256), "sweep_kernel": None}
NCU_TRAFFIC_NOTE = "bytes of the ncu captures in profiles/ (1024 tables) and, for each table more, its 13 B per cell and its share of the bytes read"
FALLBACK_HBM_GBS = 6650.0


def make_workload(name: str, scale: str, rank: int):
    if name == "cfg4":
        if scale == "small":
            return wl.config4(n_tables=256, seed_offset=1000 * rank)
        if scale == "quarter":
            return wl.config4(n_tables=1024, seed_offset=1000 * rank)
        return wl.config4(seed_offset=1000 * rank)
    if name == "cfg3":
        if scale == "small":
            return wl.config3(n_m=8, m_lo=256 << 10, m_hi=2 << 20, s_hi=256 << 10)
        return wl.config3()
    if name == "cfg2":
        return wl.config2()
    if name == "cfg5":
        return wl.config5()
    if name == "cfg1":
        return wl.config1()
    raise SystemExit("unknown workload %s" % name)


def work_counts(w):
    """Cells of one step and the algorithmic work of each kernel, in issue slots of a 64-lane pipe (the FP64 pipe's
    measured rate is the peak).  Candidates of the segmented strategies are ruled out for ranges of process counts, or many
    at a time, and cost nothing per cell then; what is counted is one DFMA per cell and strategy with lines in P, its
    winner's.  Models that depend on floor and ceil of log2 P alone (ids 6 to 9) have the same value for all process counts
    in between: not counted as slots in decide_kernel and segmin_kernel.  Elsewhere an unsegmented cell is one DFMA, a Scatter Chain
    element one interpolation DFMA, one running-sum DADD and the model's DFMA.  HBM bytes are the decision table written once
    (13 B per decision cell).  model_cells stays the number of (strategy, P, m, s) cells that the question has, whose minima are
    found: it says how fast the question is answered, not what is evaluated."""
    mask = w.strategy_mask
    seg_ids = [b for b in (2, 5, 9) if (mask >> b) & 1]
    unseg_b = [b for b in (0, 1, 3, 4, 6, 7, 8) if (mask >> b) & 1]
    scat = [b for b in (10, 11, 12) if (mask >> b) & 1]
    cells_pm = w.n_tables * w.n_P * w.n_m
    seg_cells = w.n_tables * w.n_P * len(seg_ids) * int(w.n_candidates().sum())
    bcast_dec = cells_pm if (seg_ids or unseg_b) else 0
    scat_dec = cells_pm if scat else 0
    line_slots = cells_pm * sum((mask >> b) & 1 for b in (2, 5))
    line_unseg = cells_pm * sum((mask >> b) & 1 for b in (0, 1, 3, 4))
    scat_slots = cells_pm * (((mask >> 10) & 1) + 3 * ((mask >> 11) & 1) + ((mask >> 12) & 1))
    long_lists = bool(seg_ids) and len(w.s_values()) > 64
    per_kernel = {}
    if long_lists:
        per_kernel["sweep_kernel"] = {"fp64_slots": cells_pm * len(seg_ids), "hbm_bytes": 0}
        per_kernel["fused_kernel"] = {"fp64_slots": len(unseg_b) * cells_pm + scat_slots, "hbm_bytes": 13 * (bcast_dec + scat_dec)}
    else:
        if seg_ids:
            per_kernel["decide_kernel"] = {"fp64_slots": line_slots + line_unseg, "hbm_bytes": 13 * bcast_dec}
            if scat:
                per_kernel["scatter_kernel"] = {"fp64_slots": scat_slots, "hbm_bytes": 13 * scat_dec}
        elif unseg_b:
            per_kernel["fused_kernel"] = {"fp64_slots": len(unseg_b) * cells_pm + scat_slots, "hbm_bytes": 13 * (bcast_dec + scat_dec)}
        elif scat:
            per_kernel["scatter_kernel"] = {"fp64_slots": scat_slots, "hbm_bytes": 13 * scat_dec}
    total_slots = sum(k["fp64_slots"] for k in per_kernel.values())
    return {"line_slots": line_slots, "model_cells": seg_cells + (len(unseg_b) + len(scat)) * cells_pm, "segmented_cells": seg_cells,
            "decision_cells": bcast_dec + scat_dec, "fp64_slots": total_slots, "hbm_bytes": 13 * (bcast_dec + scat_dec),
            "per_kernel": per_kernel}


class ClockSampler:
    """Samples SM clock, power and throttle reasons of one GPU through NVML while a region runs."""

    def __init__(self, uuid: str, period_s: float = 0.02):
        self.samples, self._stop, self._thread, self.sm_max, self.err = [], threading.Event(), None, None, None
        try:
            import pynvml
            pynvml.nvmlInit()
            self.nv = pynvml
            self.h = pynvml.nvmlDeviceGetHandleByUUID(uuid.encode() if hasattr(uuid, "encode") else uuid)
            self.sm_max = pynvml.nvmlDeviceGetMaxClockInfo(self.h, pynvml.NVML_CLOCK_SM)
        except Exception as e:  # NVML missing: report it instead of clocks
            self.nv, self.err = None, repr(e)
        self.period = period_s

    def _run(self):
        nv = self.nv
        while not self._stop.is_set():
            try:
                self.samples.append((nv.nvmlDeviceGetClockInfo(self.h, nv.NVML_CLOCK_SM),
                                     nv.nvmlDeviceGetPowerUsage(self.h) / 1000.0,
                                     nv.nvmlDeviceGetCurrentClocksEventReasons(self.h)))
            except Exception as e:
                self.err = repr(e)
                return
            time.sleep(self.period)

    def __enter__(self):
        if self.nv:
            self._thread = threading.Thread(target=self._run, daemon=True)
            self._thread.start()
        return self

    def __exit__(self, *exc):
        self._stop.set()
        if self._thread:
            self._thread.join()

    def summary(self):
        if not self.samples:
            return {"sm_mhz": None, "sm_max_mhz": self.sm_max, "reasons": [], "error": self.err or "no samples"}
        nv = self.nv
        names = {"sw_power_cap": nv.nvmlClocksEventReasonSwPowerCap, "hw_slowdown": nv.nvmlClocksEventReasonHwSlowdown,
                 "hw_thermal_slowdown": nv.nvmlClocksEventReasonHwThermalSlowdown,
                 "sw_thermal_slowdown": nv.nvmlClocksEventReasonSwThermalSlowdown,
                 "hw_power_brake": nv.nvmlClocksEventReasonHwPowerBrakeSlowdown}
        seen = 0
        for _, _, r in self.samples:
            seen |= r
        return {"sm_mhz": statistics.median(s[0] for s in self.samples), "sm_max_mhz": self.sm_max,
                "reasons": [k for k, bit in names.items() if seen & bit],
                "power_w_max": max(s[1] for s in self.samples), "samples": len(self.samples)}


def max_over_ranks(value: float, world: int, device) -> float:
    """Largest value over all ranks (timings of a multi-GPU run are the slowest rank's)."""
    if world == 1:
        return float(value)
    import torch
    import torch.distributed as dist
    t = torch.tensor([value], dtype=torch.float64, device=device)
    dist.all_reduce(t, op=dist.ReduceOp.MAX)
    return float(t.item())


def measured_peaks():
    p = os.path.join(ROOT, "MEASURED_PEAKS.json")
    if os.path.exists(p):
        return json.load(open(p)).get("hbm_gbs", FALLBACK_HBM_GBS), "measured"
    return FALLBACK_HBM_GBS, "fallback"


def _omp_set_threads(n: int) -> None:
    """Thread count of the OpenMP runtime the oracle's shared object runs on (the oracle itself is untouched)."""
    import ctypes
    ctypes.CDLL("libgomp.so.1").omp_set_num_threads(int(n))


def oracle_sample_rate(w, budget_s: float, threads: int = 0):
    """Times the CPU oracle, as it stands, on a bounded sample of the workload: whole tables for the
    multi-table workload, otherwise a strided subset of the process counts.  threads = 0 keeps all host
    cores, 1 times a single thread.  -> (cells/s, cores, text)."""
    from oracle import plogp_oracle as po
    all_threads = po.threads()
    if threads:
        _omp_set_threads(threads)
    try:
        return _oracle_sample_rate(po, w, budget_s)
    finally:
        if threads:
            _omp_set_threads(all_threads)


def _oracle_sample_rate(po, w, budget_s: float):
    sg = po.SGrid(w.s_list) if w.s_list is not None else po.SGrid(lo=w.s_lo, hi=w.s_hi, step=w.s_step)
    per_table_cells = w.model_cells() / w.n_tables

    def run_tables(n):
        t0 = time.perf_counter()
        for t in range(n):
            tab = po.Table(w.table_sizes(t), w.gaps[t], w.latency[t])
            po.select_grid(w.strategy_mask, po.predict_grid(tab, w.strategy_mask, w.P_values(), w.m, sg, w.k_mode))
        return time.perf_counter() - t0

    def run_stride(stride):
        P = w.P_values()[::stride]
        tab = po.Table(w.table_sizes(0), w.gaps[0], w.latency[0])
        t0 = time.perf_counter()
        po.select_grid(w.strategy_mask, po.predict_grid(tab, w.strategy_mask, P, w.m, sg, w.k_mode))
        return time.perf_counter() - t0, per_table_cells * len(P) / w.n_P

    if w.n_tables > 1:
        t1 = run_tables(1)
        n = int(max(1, min(w.n_tables, budget_s / max(t1, 1e-6))))
        dt = run_tables(n)
        return n * per_table_cells / dt, po.threads(), "first %d of %d tables, full P x m x s grid" % (n, w.n_tables)
    stride = max(1, w.n_P // 8)
    dt, cells = run_stride(stride)
    while dt < budget_s / 4 and stride > 1:
        stride = max(1, int(stride / min(4.0, budget_s / max(dt, 1e-6))))
        dt, cells = run_stride(stride)
    return cells / dt, po.threads(), "every %d-th process count of table 0, all m and s" % stride


def run_reference(args, rank):
    """The reference arm: there is no reference implementation, so this times the CPU oracle, as it
    stands, on a bounded sample of the workload (rank 0 only)."""
    if rank != 0:
        return
    w = make_workload(args.workload, args.scale, 0)
    budget = args.reference_budget / max(1, args.steps + args.warmup)
    rates, text, cores = [], "", 1
    for i in range(args.warmup + args.steps):
        r, cores, text = oracle_sample_rate(w, min(20.0, budget))
        if i >= args.warmup:
            rates.append(r)
    value = statistics.mean(rates)
    print(json.dumps({
        "impl": "reference", "metric": "model_cells_per_sec", "value": value, "unit": "cells/s", "n_gpus": args.gpus,
        "steps": args.steps, "warmup": args.warmup, "ms_per_step": 1e3 * w.model_cells() / value,
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "config": {"workload": w.name, "call": "plogp_predict" if args.call == "predict" else "plogp_select_best",
                   "note": "CPU oracle on a bounded sample; ms_per_step extrapolates to the full step"},
        "cpu_baseline": {"value": value, "unit": "cells/s", "cores": cores, "kind": "oracle", "sample": text},
        "e2e": {"value": value, "unit": "cells/s", "h2d_bytes_per_step": 0, "d2h_bytes_per_step": 0},
        "gpu_launches": 0}))


def predict_counts(w, counts):
    """Work of plogp_predict on a workload: the same model cells, but every enabled plane is written out
    (8 B per cell, plus 4 B per cell for the best segment size of each segmented strategy).  Short candidate
    lists: segmin_kernel evaluates the segmented cells and writes their planes, fused_kernel the rest."""
    n_on = bin(w.strategy_mask).count("1")
    n_seg = sum((w.strategy_mask >> b) & 1 for b in (2, 5, 9))
    cells_pm = w.n_tables * w.n_P * w.n_m
    out_bytes = cells_pm * (8 * n_on + 4 * n_seg)
    seg_bytes = cells_pm * 12 * n_seg
    unseg = n_on - n_seg + 2 * ((w.strategy_mask >> 11) & 1)  # the closed-form planes, in FP64
    c = dict(counts)
    if "sweep_kernel" in counts["per_kernel"]:
        sweep = counts["per_kernel"]["sweep_kernel"]
        c["per_kernel"] = {"sweep_kernel": sweep, "fused_kernel": {"fp64_slots": unseg * cells_pm, "hbm_bytes": out_bytes}}
    elif n_seg:
        c["per_kernel"] = {"segmin_kernel": {"fp64_slots": counts["line_slots"], "hbm_bytes": seg_bytes},
                           "fused_kernel": {"fp64_slots": unseg * cells_pm, "hbm_bytes": out_bytes - seg_bytes}}
    else:
        c["per_kernel"] = {"fused_kernel": {"fp64_slots": unseg * cells_pm, "hbm_bytes": out_bytes}}
    c["fp64_slots"] = sum(k["fp64_slots"] for k in c["per_kernel"].values())
    c["hbm_bytes"] = out_bytes
    return c


class Bench:
    """One rank's measuring context: device, process group, peaks."""

    def __init__(self, rank, local_rank, world):
        import torch
        from paper_cs_0408034_b200 import plogp
        self.torch, self.plogp = torch, plogp
        self.rank, self.local_rank, self.world = rank, local_rank, world
        self.dist = None
        torch.cuda.set_device(local_rank)
        if world > 1:
            import torch.distributed as dist
            dist.init_process_group("nccl", device_id=torch.device("cuda", local_rank))
            self.dist = dist
        self.flush_buf = None
        self.fma_rate = None
        self.hbm_gbs, self.peak_src = measured_peaks()

    def barrier(self):
        if self.dist is not None:
            self.dist.barrier()
        self.torch.cuda.synchronize()

    def close(self):
        if self.dist is not None:
            self.dist.destroy_process_group()

    def time_device(self, w, predict, steps, warmup, clocks_uuid=None):
        """Device-resident timing of `steps` steps of one call on one workload.  Returns the measured
        dictionary; the per-kernel times come from a few more steps in which the library records events around each
        launch (its kernels do not overlap then, so they add up to a little more than a step)."""
        torch, plogp = self.torch, self.plogp
        counts = work_counts(w)
        grid = plogp.GridArgs.from_workload(w)
        tabs = plogp.Tables.from_workload(w)
        if predict:
            counts = predict_counts(w, counts)
            out = plogp.predict(tabs, grid)
            out_bytes = counts["hbm_bytes"]
        else:
            out = plogp.alloc_decision(w.n_tables, w.n_P, w.n_m)
            out_bytes = out.strategy.numel() * 13
        flush = None
        if out_bytes < (256 << 20):  # outputs do not evict the 126 MB L2 by themselves: write 256 MB between steps
            if self.flush_buf is None:
                self.flush_buf = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
            flush = self.flush_buf

        def step():
            if predict:
                plogp.predict(tabs, grid, out=out)
            else:
                plogp.select_best(tabs, grid, out=out)

        for _ in range(warmup):
            step()
            if flush is not None:
                flush.fill_(1)
        self.barrier()
        launches0 = plogp.kernel_launches()
        events = [(torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)) for _ in range(steps)]
        with ClockSampler(clocks_uuid) as clocks:
            self.barrier()
            for a, b in events:
                a.record()
                step()
                b.record()
                if flush is not None:
                    flush.fill_(1)
            self.barrier()
        launches = plogp.kernel_launches() - launches0
        kernel_steps = max(3, min(steps, 10))
        plogp.profile_enable(tabs, True)
        for _ in range(kernel_steps):
            step()
            if flush is not None:
                flush.fill_(1)
        kernel_ms = plogp.profile_read(tabs)   # {kernel: (ms over these steps, launches)}
        plogp.profile_enable(tabs, False)
        total_ms = max_over_ranks(sum(a.elapsed_time(b) for a, b in events), self.world, "cuda")
        return {"w": w, "predict": predict, "counts": counts, "steps": steps, "ms_per_step": total_ms / steps, "launches": launches,
                "kernel_ms": kernel_ms, "kernel_steps": kernel_steps, "out_bytes": out_bytes, "flushed": flush is not None, "clocks": clocks,
                "tabs": tabs, "grid": grid}

    def time_e2e(self, m, steps):
        """The same step through the public API with HOST buffers: the host tables go in
        (plogp_table_update) and the decision table comes back into page-locked host arrays
        (plogp_select_best_host); every copy is inside the timed region."""
        plogp, w, tabs, grid = self.plogp, m["w"], m["tabs"], m["grid"]
        host = plogp.alloc_decision_host(w.n_tables, w.n_P, w.n_m)
        h2d = w.sizes.nbytes + w.gaps.nbytes + w.latency.nbytes + w.m.nbytes + (0 if w.s_list is None else w.s_list.nbytes)
        d2h = sum(t.numel() * t.element_size() for t in (host.strategy, host.s_bytes, host.time))

        def e2e_step():
            tabs.update(w.sizes, w.gaps, w.latency)
            plogp.select_best_host(tabs, grid, out=host)

        e2e_step()
        self.barrier()
        t0 = time.perf_counter()
        for _ in range(steps):
            e2e_step()
        self.barrier()
        ms = max_over_ranks((time.perf_counter() - t0) * 1e3 / steps, self.world, "cuda")
        return ms, h2d, d2h

    def time_aux(self, name, w, fn, nbytes, steps=10, warmup=3):
        """Times one streaming call (CUDA events on the launching stream, L2 flushed between steps when the
        call moves less than 256 MB) and reports it against the HBM roofline of its algorithmic bytes."""
        torch = self.torch
        if self.flush_buf is None:
            self.flush_buf = torch.empty(256 << 20, dtype=torch.uint8, device="cuda")
        flush = nbytes < (256 << 20)
        for _ in range(warmup):
            fn()
        torch.cuda.synchronize()
        ms = 0.0
        for _ in range(steps):
            if flush:
                self.flush_buf.fill_(1)
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            fn()
            b.record()
            b.synchronize()
            ms += a.elapsed_time(b)
        ms /= steps
        return {"call": name, "config": {"workload": w.name, "tables_per_gpu": w.n_tables, "P": [w.P_lo, w.P_hi], "n_m": w.n_m,
                                         "n_s": int(len(w.s_values()))},
                "steps": steps, "ms_per_step": ms,
                "roofline": {"bound": "hbm", "achieved": nbytes / (ms * 1e-3) / 1e9, "peak": self.hbm_gbs, "unit": "GB/s",
                             "frac": nbytes / (self.hbm_gbs * 1e9) / (ms * 1e-3), "algorithmic_bytes": nbytes,
                             "peak_source": "HBM copy bandwidth, of %s" % self.peak_src}}

    def graph_entries(self):
        """The launch-bound grids again, replayed from a captured CUDA graph: with its plan cached a call only
        launches kernels on the caller's stream, so a loop of calls can be captured once and replayed.  Back-to-back
        calls (no L2 flush between them), device time per call, next to the same loop of direct calls."""
        plogp, torch = self.plogp, self.torch
        out = []
        for w in (wl.config1(), wl.config2(), wl.config5()):
            with plogp.Tables.from_workload(w) as tabs:
                g = plogp.GridArgs.from_workload(w)
                dec = plogp.select_best(tabs, g)  # builds the plan, allocates scratch
                torch.cuda.synchronize()
                st = torch.cuda.Stream()
                graph = torch.cuda.CUDAGraph()
                with torch.cuda.stream(st):
                    plogp.select_best(tabs, g, out=dec, stream=st)
                    st.synchronize()
                    with torch.cuda.graph(graph, stream=st):
                        plogp.select_best(tabs, g, out=dec, stream=st)
                n = 200

                def per_call(fn):
                    for _ in range(10):
                        fn()
                    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                    a.record()
                    for _ in range(n):
                        fn()
                    b.record()
                    b.synchronize()
                    return a.elapsed_time(b) / n
                t_graph = per_call(graph.replay)
                t_direct = per_call(lambda: plogp.select_best(tabs, g, out=dec))
                out.append({"workload": w.name, "calls": n, "ms_per_call_graph_replay": t_graph, "ms_per_call_direct": t_direct,
                            "note": "back-to-back calls, no L2 flush"})
                del graph
        return out

    def aux_entries(self, w4):
        """The segment-size sensitivity calls: the model surface over s on the dense single-table grid, the fixed
        8 kB segment size and the decision boundaries on the batched workload."""
        plogp, torch = self.plogp, self.torch
        out = []
        w2 = wl.config2()
        with plogp.Tables.from_workload(w2) as tabs:
            g = plogp.GridArgs.from_workload(w2)
            surf = plogp.segment_surface(tabs, g)
            out.append(self.time_aux("plogp_segment_surface", w2, lambda: plogp.segment_surface(tabs, g, out=surf), surf.numel() * 8))
            del surf
        with plogp.Tables.from_workload(w4) as tabs:
            g = plogp.GridArgs.from_workload(w4)
            pred = plogp.predict(tabs, g)
            cells = w4.n_tables * w4.n_P * w4.n_m
            shape = (w4.n_tables, 3, w4.n_P, w4.n_m)
            fixed = torch.empty(shape, dtype=torch.float64, device="cuda")
            ratio = torch.empty(shape, dtype=torch.float64, device="cuda")

            def sens():
                plogp._check(plogp.lib.plogp_segment_sensitivity(tabs.handle, g.ref, 8192, pred.time.data_ptr(), fixed.data_ptr(),
                                                                 ratio.data_ptr(), plogp._stream_ptr(None)), "plogp_segment_sensitivity")
            out.append(self.time_aux("plogp_segment_sensitivity (s = 8192 B)", w4, sens, 3 * cells * 8 * 3))
            del pred, fixed, ratio
            dec = plogp.select_best(tabs, g)
            bnd = torch.empty_like(dec.strategy)

            def bounds():
                plogp._check(plogp.lib.plogp_decision_boundaries(w4.n_tables, w4.n_P, w4.n_m, dec.strategy.data_ptr(), bnd.data_ptr(),
                                                                 plogp._stream_ptr(None)), "plogp_decision_boundaries")
            out.append(self.time_aux("plogp_decision_boundaries", w4, bounds, 2 * cells * 2))
        return out

    def rooflines(self, m):
        """Per-kernel roofline objects of one measurement, the dominant kernel's copy and the whole-step figure."""
        if self.fma_rate is None:
            self.fma_rate = self.plogp.fp64_fma_rate(100.0)
        fma_rate, hbm_gbs = self.fma_rate, self.hbm_gbs
        counts, steps, w = m["counts"], m["kernel_steps"], m["w"]

        def roof(name, ms_total, n_launch):
            # algorithmic work per launch / average launch duration (CUDA events recorded by the library on
            # the launching stream)
            work = counts["per_kernel"].get(name)
            if work is None or n_launch == 0:
                return {"kernel": name, "launches": n_launch, "ms_total": ms_total, "avg_ms": ms_total / max(n_launch, 1)}
            per_launch = steps / n_launch  # a kernel launched once per step does one step's work
            dur = ms_total / n_launch * 1e-3
            slots, nbytes = work["fp64_slots"] * per_launch, work["hbm_bytes"] * per_launch
            t_alu, t_hbm = slots / fma_rate, nbytes / (hbm_gbs * 1e9)
            alu = t_alu >= t_hbm
            r = {"kernel": name, "launches": n_launch, "ms_total": ms_total, "avg_ms": dur * 1e3,
                 "bound": "alu" if alu else "hbm",
                 "achieved": slots / dur / 1e12 if alu else nbytes / dur / 1e9,
                 "peak": fma_rate / 1e12 if alu else hbm_gbs,
                 "unit": "T slots/s of a 64-lane pipe" if alu else "GB/s",
                 "frac": max(t_alu, t_hbm) / dur,
                 "alu_time_ms": t_alu * 1e3, "hbm_time_ms": t_hbm * 1e3,
                 "peak_source": ("DFMA issue rate measured in this run by plogp_fp64_fma_rate, of measured (nominal %.2f T/s = 148 SMs x 64 lanes x 1.965 GHz)"
                                 % (NOMINAL_FP64_FMA_RATE / 1e12)) if alu else "HBM copy bandwidth, of %s" % self.peak_src}
            return r

        kernels = [roof(k, v[0], v[1]) for k, v in m["kernel_ms"].items()]
        tot = sum(k["ms_total"] for k in kernels) or 1.0
        for k in kernels:
            k["share"] = k["ms_total"] / tot
        dominant = dict(max(kernels, key=lambda k: k["ms_total"])) if kernels else {}
        captured = NCU_TRAFFIC.get(dominant.get("kernel"))
        dominant["traffic"] = None
        if captured and w.name.startswith("cfg4") and not m["predict"] and w.n_tables >= NCU_TRAFFIC_TABLES:
            read, written = captured
            per_table = read / NCU_TRAFFIC_TABLES + 13.0 * w.n_P * w.n_m
            dominant["traffic"] = read + written + (w.n_tables - NCU_TRAFFIC_TABLES) * per_table
        dominant["traffic_note"] = NCU_TRAFFIC_NOTE if dominant["traffic"] else None
        t_alu = counts["fp64_slots"] / fma_rate
        t_hbm = counts["hbm_bytes"] / (hbm_gbs * 1e9)
        dominant["step"] = {"frac": max(t_alu, t_hbm) / (m["ms_per_step"] * 1e-3), "alu_time_ms": t_alu * 1e3, "hbm_time_ms": t_hbm * 1e3,
                            "note": "whole step (all kernels) against max(issue slots, HBM bytes)"}
        return kernels, dominant

    def config_of(self, m):
        w, counts = m["w"], m["counts"]
        return {"workload": w.name, "call": "plogp_predict" if m["predict"] else "plogp_select_best", "tables_per_gpu": w.n_tables,
                "P": [w.P_lo, w.P_hi], "n_m": w.n_m, "n_s": int(len(w.s_values())), "strategy_mask": w.strategy_mask,
                "model_cells_per_gpu": counts["model_cells"], "decision_cells_per_gpu": counts["decision_cells"],
                "parallelism": "tables sharded, %d rank(s)" % self.world,
                "evaluation": "candidates ruled out by bounds over ranges of process counts (short lists) or groups of sizes (long ones), the "
                              "rest evaluated in FP64; ids 6 to 9 once per (floor, ceil) of log2 P; results are those of the exhaustive "
                              "FP64 search; model cells are those of the question, evaluated or ruled out",
                "l2": "256 MB written between timed steps to flush L2" if m["flushed"]
                else "outputs (%.1f GB per step) exceed the 126 MB L2" % (m["out_bytes"] / 1e9)}

    def entry(self, m, note=None):
        """One element of the `workloads` list."""
        step_s = m["ms_per_step"] * 1e-3
        if getattr(m["w"], "search_mode", 0) == 1:
            # lower-envelope search: most (P, m, s) cells are never visited, so no model-cell rate and no
            # roofline against the exhaustive work; decision cells per second and the kernel times are what counts
            cfg = self.config_of(m)
            cfg["search_mode"] = 1
            cfg.pop("model_cells_per_gpu")
            e = {"config": cfg, "steps": m["steps"], "ms_per_step": m["ms_per_step"], "model_cells_per_sec": None,
                 "decision_cells_per_sec": m["counts"]["decision_cells"] / step_s,
                 "gpu_launches_per_step": m["launches"] / m["steps"],
                 "kernels": [{"kernel": k, "launches": v[1], "avg_ms": v[0] / v[1]} for k, v in m["kernel_ms"].items()]}
        else:
            kernels, dominant = self.rooflines(m)
            e = {"config": self.config_of(m), "steps": m["steps"], "ms_per_step": m["ms_per_step"],
                 "model_cells_per_sec": m["counts"]["model_cells"] / step_s, "decision_cells_per_sec": m["counts"]["decision_cells"] / step_s,
                 "gpu_launches_per_step": m["launches"] / m["steps"], "roofline": dominant}
        if note:
            e["note"] = note
        return e


def _free(m):
    m["tabs"].free()
    m.pop("tabs"); m.pop("grid")


def run_ours(args, rank, local_rank, world):
    if args.warmup < 3:
        args.warmup = 3
    b = Bench(rank, local_rank, world)
    torch = b.torch
    uuid = str(torch.cuda.get_device_properties(local_rank).uuid)
    if not uuid.startswith("GPU-"):
        uuid = "GPU-" + uuid

    w = make_workload(args.workload, args.scale, rank)
    if args.search == "envelope":
        from dataclasses import replace as _replace
        w = _replace(w, search_mode=1)
    predict = args.call == "predict"
    m = b.time_device(w, predict, args.steps, args.warmup, clocks_uuid=uuid)
    e2e_ms, h2d, d2h = None, 0, 0
    if args.e2e_steps > 0 and not predict:
        e2e_ms, h2d, d2h = b.time_e2e(m, args.e2e_steps)
    _free(m)
    if rank != 0:
        b.close()
        return

    kernels, roofline = b.rooflines(m)
    counts, step_s = m["counts"], m["ms_per_step"] * 1e-3
    if args.search == "envelope":
        # most cells are never visited: report decision cells, and no roofline against the exhaustive work
        print(json.dumps({"metric": "decision_cells_per_sec", "value": world * counts["decision_cells"] / step_s, "unit": "cells/s",
                          "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "ms_per_step": m["ms_per_step"],
                          "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
                          "config": dict(b.config_of(m), search_mode=1), "clocks": m["clocks"].summary(), "gpu_launches": m["launches"],
                          "kernels": [{"kernel": k, "launches": v[1], "avg_ms": v[0] / v[1]} for k, v in m["kernel_ms"].items()]}))
        b.close()
        return
    line = {
        "metric": "model_cells_per_sec", "value": world * counts["model_cells"] / step_s, "unit": "cells/s",
        "n_gpus": world, "steps": args.steps, "warmup": args.warmup, "ms_per_step": m["ms_per_step"],
        "higher_is_better": True, "scaling": "weak", "vs_baseline": None, "dtype": "f64", "data": "synthetic",
        "decision_cells_per_sec": world * counts["decision_cells"] / step_s,
        "config": b.config_of(m),
        "clocks": m["clocks"].summary(),
        "e2e": {"value": None if e2e_ms is None else world * counts["model_cells"] / (e2e_ms * 1e-3), "unit": "cells/s",
                "ms_per_step": e2e_ms, "steps": args.e2e_steps, "h2d_bytes_per_step": h2d, "d2h_bytes_per_step": d2h},
        "gpu_launches": m["launches"],
        "roofline": roofline,
        "kernels": kernels,
    }
    if world == 1 and not args.no_workloads and args.workload == "cfg4" and args.scale == "full" and not predict:
        # the other configurations, in the same run: fewer steps, same timing rules
        others = []
        k = max(3, min(args.steps, 10))
        mm = b.time_device(wl.config3(), False, k, 3)
        _free(mm)
        others.append(b.entry(mm))
        mm = b.time_device(w, True, k, 3)
        _free(mm)
        others.append(b.entry(mm))
        for make in (wl.config2, wl.config5, wl.config1):
            mm = b.time_device(make(), False, max(k, 20), 5)
            _free(mm)
            others.append(b.entry(mm, note="launch-bound: microseconds of work per call; reported, not judged against the 60 % bar"))
        from dataclasses import replace
        for base in (wl.config3(), w):
            mm = b.time_device(replace(base, search_mode=1), False, k, 3)
            _free(mm)
            others.append(b.entry(mm, note="segment search by lower envelope (search_mode 1): same decision table, "
                                           "skipped cells are not counted as model cells"))
        line["workloads"] = others
        line["sensitivity_calls"] = b.aux_entries(w)
        line["graph_replay"] = b.graph_entries()
    if world == 1 and not args.no_cpu_baseline:
        v, cores, text = oracle_sample_rate(w, 15.0)
        v1, _, text1 = oracle_sample_rate(w, 8.0, threads=1)
        line["cpu_baseline"] = {"value": v, "unit": "cells/s", "cores": cores, "kind": "oracle", "sample": text,
                                "single_thread": {"value": v1, "unit": "cells/s", "cores": 1, "sample": text1}}
    print(json.dumps(line))
    b.close()


def _spawned(local_rank, argv, world, port):
    os.environ.update(RANK=str(local_rank), LOCAL_RANK=str(local_rank), WORLD_SIZE=str(world),
                      MASTER_ADDR="127.0.0.1", MASTER_PORT=str(port))
    sys.argv = argv
    main()


def main():
    ap = argparse.ArgumentParser()
    ap.add_argument("--gpus", type=int, default=1)
    ap.add_argument("--steps", type=int, default=100)
    ap.add_argument("--warmup", type=int, default=5)
    ap.add_argument("--impl", default="ours", choices=["ours", "reference"])
    ap.add_argument("--workload", default="cfg4", choices=["cfg1", "cfg2", "cfg3", "cfg4", "cfg5"])
    ap.add_argument("--scale", default="full", choices=["full", "quarter", "small"],
                    help="quarter / small: reduced copies of the batched workload and the sweep for profiler captures")
    ap.add_argument("--e2e-steps", type=int, default=3)
    ap.add_argument("--call", default="select_best", choices=["select_best", "predict"],
                    help="predict: time plogp_predict (all model planes) instead of the decision table; device-resident only")
    ap.add_argument("--search", default="exhaustive", choices=["exhaustive", "envelope"],
                    help="envelope: plogp_grid.search_mode = 1 for the headline workload (same decision table, most cells skipped)")
    ap.add_argument("--no-cpu-baseline", action="store_true")
    ap.add_argument("--no-workloads", action="store_true", help="headline workload only (no `workloads` list)")
    ap.add_argument("--reference-budget", type=float, default=120.0, help="seconds of oracle time for --impl reference")
    args = ap.parse_args()

    if args.impl == "reference":
        run_reference(args, int(os.environ.get("RANK", "0")))
        return
    if "WORLD_SIZE" not in os.environ and args.gpus > 1:
        # started without a launcher: one process per GPU from here
        import socket
        import torch.multiprocessing as mp
        s = socket.socket()
        s.bind(("127.0.0.1", 0))
        port = s.getsockname()[1]
        s.close()
        mp.spawn(_spawned, args=(list(sys.argv), args.gpus, port), nprocs=args.gpus, join=True)
        return
    run_ours(args, int(os.environ.get("RANK", "0")), int(os.environ.get("LOCAL_RANK", "0")),
             int(os.environ.get("WORLD_SIZE", "1")))


if __name__ == "__main__":
    main()
