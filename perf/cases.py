"""What is timed when this library's speed is looked at: the calls a tuner makes, at the sizes it makes them.

A case is one pass of a tuner's program through the public calls of ``paper_cs_0408034_b200.plogp``:

  decide     ``select_best`` on short candidate lists (<= 64 segment sizes), the decision table of Broadcast and Scatter
  sweep      ``select_best`` with every multiple of 4 B as a candidate segment size
  scatter    ``select_best`` with the Scatter strategies alone, long ranges of process counts
  predict    ``predict``: every model's plane and the best segment sizes
  tune_all   the decision tables of all five collectives on one handle: ``select_best`` and the three
             ``select_best_collective`` calls
  study      how much the segment size matters: ``segment_surface`` for a few process counts,
             ``segment_sensitivity`` of the fixed 8 kB size and ``decision_boundaries`` for the whole grid
  retune     new measured tables in (``update``), decision table out into host arrays (``select_best_host``)

The grids are those of ``workloads.config1`` .. ``config5`` and of the parity tests; the tables are drawn from the
same laws with the seed that ``prepare`` is given.
"""
import math

import numpy as np
import torch

from paper_cs_0408034_b200 import plogp, workloads

ALL = workloads.ALL_STRATEGIES
ETHERNET = sum(1 << i for i in (0, 3, 5, 6, 7, 10, 11, 12))  # the strategies of workloads.config1
SEG_PAIR = (1 << 2) | (1 << 5)                               # Segmented Flat Tree and Segmented Chain
SCATTER = 7 << 10
KIB, MIB = 1 << 10, 1 << 20


def _case(name, kind, tables, P_lo, P_hi, n_P, m_lo, m_hi, n_m, s_lo, s_hi, n_s, mask, net, n_bp, k_mode=0, search=0, dips=False, fresh=False):
    """n_P = 0: every process count from P_lo to P_hi, else n_P of them, log-spaced.  n_s = 0: every multiple of 4 B.
    search: plogp_grid.search_mode.  dips: tables as measured, not forced to grow with the size.  fresh: the call makes
    its own outputs, as in the README's example."""
    named = {} if name is None else {"name": name}
    return {**named, "kind": kind, "tables": tables, "P_lo": P_lo, "P_hi": P_hi, "n_P": n_P, "m_lo": m_lo, "m_hi": m_hi, "n_m": n_m,
            "s_lo": s_lo, "s_hi": s_hi, "n_s": n_s, "mask": mask, "net": net, "n_bp": n_bp, "k_mode": k_mode, "search": search,
            "dips": dips, "fresh": fresh}


def listed():
    return [
        # The README's example: one Ethernet-like table, P = 2..50, new outputs with each call.  What a launcher asks for
        # one cluster; only latency counts.
        _case("decide_ethernet", "decide", 1, 2, 50, 0, 4, MIB, 19, KIB, 64 * KIB, 7, ETHERNET, "ethernet", 21, fresh=True),
        # One table on a dense grid, all strategies: a decision table for one network, to be kept.
        _case("decide_dense", "decide", 1, 2, 1024, 0, 4, 64 * MIB, 256, 4, MIB, 64, ALL, "ethernet", 21),
        # Batched tuning of 4096 networks: the benchmark's default workload.
        _case("decide_batched", "decide", 4096, 2, 512, 0, 4, 64 * MIB, 128, 4, MIB, 32, ALL, "mixed", 64),
        # A service that tunes a thousand networks for the process counts its users run, with the lower-envelope search;
        # odd sizes everywhere, the floor rule for the number of segments.
        _case("decide_listed_envelope", "decide", 1000, 2, 3000, 203, 4, 48 * MIB, 101, 4, MIB, 27, ALL, "mixed", 50, k_mode=1, search=1),
        # Exhaustive segment sweep: every multiple of 4 B up to 1 MB.
        _case("sweep_exhaustive", "sweep", 1, 2, 4096, 0, 4 * KIB, 16 * MIB, 128, 4, MIB, 0, SEG_PAIR, "fast", 64),
        # The same question asked with the lower-envelope search.
        _case("sweep_envelope", "sweep", 1, 2, 4096, 0, 4 * KIB, 16 * MIB, 128, 4, MIB, 0, SEG_PAIR, "fast", 64, search=1),
        # Scatter of small blocks on a large machine: sums over up to 65535 gaps.
        _case("scatter_long", "scatter", 1, 2, 65536, 0, 4, 4 * KIB, 64, 4, 4, 0, SCATTER, "fast", 128),
        # Every model's prediction for one measured network (the table as measured, dips and all); ragged sizes.
        _case("predict_measured", "predict", 1, 3, 1001, 0, 4, 64 * MIB, 255, 4, MIB, 63, ALL, "ethernet", 41, dips=True),
        # Predictions for a batch of networks: 7.8 GB of planes.
        _case("predict_batched", "predict", 1024, 2, 512, 0, 4, 64 * MIB, 128, 4, MIB, 32, ALL, "mixed", 64),
        # The tables of all five collectives for a batch of networks, on one handle.
        _case("tune_all_collectives", "tune_all", 64, 2, 512, 0, 4, 64 * MIB, 128, 4, MIB, 32, ALL, "mixed", 64),
        # How much the segment size matters, over a batch of networks.
        _case("segment_study", "study", 256, 2, 512, 0, 4, 64 * MIB, 128, 4, MIB, 32, ALL, "mixed", 64),
        # A tuner that follows its networks: new tables from the host, decision table back into page-locked host arrays.
        _case("retune_to_host", "retune", 64, 2, 512, 0, 4, 64 * MIB, 128, 4, MIB, 32, ALL, "mixed", 64),
    ]


def _log_int(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(("decide", "decide", "decide", "sweep", "scatter", "predict", "predict", "tune_all", "study", "retune"))
    net = rng.choice(("ethernet", "mixed", "mixed", "fast"))
    n_bp = _log_int(rng, 12, 200)
    k_mode = int(rng.random() < 0.25)
    dips = rng.random() < 0.25
    search = int(rng.random() < 0.3)
    if kind == "scatter":
        P_hi = _log_int(rng, 1000, 65536)
        return _case(None, kind, _log_int(rng, 1, 8), rng.choice((2, 2, 7)), P_hi, 0, 4, _log_int(rng, 256, 4 * KIB), _log_int(rng, 8, 64),
                     4, 4, 0, SCATTER, net, n_bp, dips=dips)
    if kind == "sweep":
        P_hi, n_m = _log_int(rng, 64, 4096), _log_int(rng, 8, 128)
        mask = rng.choice((SEG_PAIR, SEG_PAIR, SEG_PAIR | (1 << 9), ALL))
        s_hi = _log_int(rng, 16, 256) * KIB
        tables = max(1, min(_log_int(rng, 1, 4), 140_000_000_000 // (3 * P_hi * n_m * s_hi // 4)))
        return _case(None, kind, tables, 2, P_hi, 0, 4 * KIB, _log_int(rng, 256, 16 * KIB) * KIB, n_m, 4, s_hi, 0, mask, net, n_bp, k_mode, search)
    P_hi = _log_int(rng, 16, 3000)
    span = P_hi - 1
    n_P = rng.choice((0, 0, min(span, _log_int(rng, 8, 300))))
    n_m, n_s = _log_int(rng, 5, 256), _log_int(rng, 4, 64)
    mask = rng.choice((ALL, ALL, ALL, ETHERNET))
    most = {"decide": 200_000_000, "predict": 60_000_000, "tune_all": 10_000_000, "study": 20_000_000, "retune": 6_000_000}[kind]
    rows = (n_P or span) * n_m
    tables = max(1, min(_log_int(rng, 1, 4096), most // rows))
    fresh = kind == "decide" and tables * rows < 1_000_000 and rng.random() < 0.5
    if kind not in ("decide", "predict", "retune"):
        search = 0
    return _case(None, kind, tables, 2, P_hi, n_P, 4, _log_int(rng, MIB, 64 * MIB), n_m, 4, _log_int(rng, 64 * KIB, MIB), n_s, mask, net, n_bp,
                 k_mode, search, dips, fresh)


def _tables(case, seed):
    """(sizes, gaps, latency) of the case's networks: the laws of workloads.config1 (ethernet), config4 (mixed) and
    config3 / config5 (fast), with noise drawn from the seed."""
    rng = np.random.default_rng(seed)
    n, n_bp, net = case["tables"], case["n_bp"], case["net"]
    top = {"ethernet": MIB, "mixed": 256 * MIB, "fast": 256 * MIB}[net]
    sizes = workloads.log_spaced_multiples(1 if net == "ethernet" else 4, top, n_bp, 1 if net == "ethernet" else 4)
    if net == "ethernet":
        latency, overhead, per_byte, eps = 50.0 * rng.uniform(0.9, 1.1, n), np.full(n, 30.0), np.full(n, 0.08), 0.02
    elif net == "fast":
        latency, overhead, per_byte, eps = rng.uniform(2.0, 5.0, n), np.full(n, 1.0), 10.0 ** rng.uniform(-4.4, -3.1, n), 0.01
    else:
        latency = workloads.log_uniform(1.0, 100.0, rng.random(n))
        overhead = workloads.log_uniform(0.5, 50.0, rng.random(n))
        per_byte = 8.0 / workloads.log_uniform(100.0, 400000.0, rng.random(n))
        eps = 0.03
    g = (overhead[:, None] + per_byte[:, None] * sizes.astype(np.float64)[None, :]) * rng.uniform(1.0 - eps, 1.0 + eps, (n, n_bp))
    if case["dips"]:
        g[:, -1] = np.maximum(g[:, -1], g[:, -2])  # the library continues the last line and asks that it does not fall
    else:
        g = np.maximum.accumulate(g, axis=1)
    return sizes, np.ascontiguousarray(g), np.ascontiguousarray(latency)


def _process_counts(case):
    """Listed process counts, or None for the whole range."""
    if not case["n_P"]:
        return None
    P = np.unique(np.rint(case["P_lo"] * (case["P_hi"] / case["P_lo"]) ** (np.arange(case["n_P"]) / max(1, case["n_P"] - 1))).astype(np.int64))
    rest = np.setdiff1d(np.arange(case["P_lo"], case["P_hi"] + 1), P)  # the short end of a logarithmic list repeats itself
    return np.sort(np.concatenate([P, rest[: case["n_P"] - len(P)]])).astype(np.int32)


def _segment_sizes(case):
    return workloads.log_spaced_multiples(case["s_lo"], case["s_hi"], case["n_s"]) if case["n_s"] else None


def _message_sizes(case):
    return workloads.log_spaced_multiples(case["m_lo"], case["m_hi"], case["n_m"])


def _grid(case, P=None):
    P = _process_counts(case) if P is None else P
    s = _segment_sizes(case)
    step = {} if s is not None else {"s_lo": case["s_lo"], "s_hi": case["s_hi"] // 4 * 4, "s_step": 4}
    return plogp.GridArgs(_message_sizes(case), P, case["P_lo"], case["P_hi"], s, strategy_mask=case["mask"], k_mode=case["k_mode"],
                          search_mode=case["search"], **step)


def _few_process_counts(case):
    return np.unique(np.array([case["P_lo"], max(case["P_lo"], case["P_hi"] // 8), case["P_hi"]], dtype=np.int32))


def prepare(case, seed):
    sizes, gaps, latency = _tables(case, seed)
    st = {"case": case, "tables": plogp.Tables(sizes, gaps, latency), "grid": _grid(case)}
    tabs, grid, kind = st["tables"], st["grid"], case["kind"]
    if kind in ("decide", "sweep", "scatter", "tune_all"):
        st["out"] = None if case["fresh"] else plogp.alloc_decision(tabs.n_tables, grid.n_P, grid.n_m)
    elif kind == "predict":
        shape = (tabs.n_tables, plogp.N_STRATEGIES, grid.n_P, grid.n_m)
        st["out"] = plogp.Prediction(torch.zeros(shape, dtype=torch.float64, device="cuda"),
                                     torch.zeros((tabs.n_tables, 3, grid.n_P, grid.n_m), dtype=torch.int32, device="cuda"))
    elif kind == "study":
        st["few"] = _grid(case, _few_process_counts(case))
        st["pred"] = plogp.predict(tabs, grid)
        st["dec"] = plogp.select_best(tabs, grid)
    else:
        st["host"] = (sizes, gaps, latency)
        st["out"] = plogp.alloc_decision_host(tabs.n_tables, grid.n_P, grid.n_m)
        for t in (st["out"].strategy, st["out"].s_bytes, st["out"].time):
            t.zero_()
    return st


def _planes(case, d):
    """The planes that the call writes (a collective without an enabled strategy has none)."""
    if case["kind"] == "scatter":
        return d.strategy[:, 1], d.s_bytes[:, 1], d.time[:, 1]
    if not case["mask"] & SCATTER:
        return d.strategy[:, 0], d.s_bytes[:, 0], d.time[:, 0]
    return d.strategy, d.s_bytes, d.time


def run(st):
    case, tabs, grid, kind = st["case"], st["tables"], st["grid"], st["case"]["kind"]
    if kind in ("decide", "sweep", "scatter"):
        return _planes(case, plogp.select_best(tabs, grid, out=st["out"]))
    if kind == "predict":
        p = plogp.predict(tabs, grid, out=st["out"])
        if case["mask"] == ALL:
            return p.time, p.best_s
        on = [i for i in range(plogp.N_STRATEGIES) if (case["mask"] >> i) & 1]
        return [p.time[:, i] for i in on] + [p.best_s[:, j] for j, i in enumerate(plogp.SEGMENTED_IDS) if i in on]
    if kind == "tune_all":
        got = list(_planes(case, plogp.select_best(tabs, grid, out=st["out"])))
        for collective in (plogp.GATHER, plogp.REDUCE, plogp.BARRIER):
            d = plogp.select_best_collective(tabs, grid, collective)
            got += [d.strategy, d.s_bytes, d.time]
        return got
    if kind == "study":
        surface = plogp.segment_surface(tabs, st["few"])
        fixed, ratio = plogp.segment_sensitivity(tabs, grid, 8 * KIB, pred=st["pred"])
        return surface, fixed, ratio, plogp.decision_boundaries(st["dec"])
    tabs.update(*st["host"])
    return _planes(case, plogp.select_best_host(tabs, grid, out=st["out"]))


def work(case):
    """Bytes: the tables and the grid in once, every written plane out once (and, in a study, the planes it reads).
    Operations: two for every (P, m, s) cell of an exhaustive search and for every unsegmented cell, four for a step of
    the Scatter Chain sum; the lower-envelope search needs one cell per (P, m) and segmented strategy."""
    mask, n_t = case["mask"], case["tables"]
    n_P = case["n_P"] or case["P_hi"] - case["P_lo"] + 1
    n_m, m = case["n_m"], _message_sizes(case)
    s = _segment_sizes(case)
    if s is None:
        s = np.arange(case["s_lo"], case["s_hi"] // 4 * 4 + 1, 4, dtype=np.uint64)
    cand = float(np.maximum(np.searchsorted(s, m, side="right"), 1).sum())  # candidates over all message sizes
    segs = [i for i in plogp.SEGMENTED_IDS if (mask >> i) & 1]
    n_on = bin(mask).count("1")
    cells = float(n_t) * n_P * n_m
    bcast, scat = bool(mask & 0x3FF), bool(mask & SCATTER)
    table_in = n_t * (case["n_bp"] * 8.0 + 8.0) + case["n_bp"] * 8.0 + n_m * 8.0 + (case["n_P"] or 0) * 4.0 + (case["n_s"] or 0) * 8.0

    def model_ops(on):
        seg = sum((on >> i) & 1 for i in segs)
        searched = 2.0 * n_t * n_P * cand * seg if case["search"] == 0 else 2.0 * cells * seg
        plain = bin(on).count("1") - seg
        return searched + 2.0 * cells * plain + (2.0 * cells if (on >> 11) & 1 else 0.0)

    kind = case["kind"]
    if kind == "predict":
        return {"bytes": table_in + cells * (8 * n_on + 4 * len(segs)), "flops": model_ops(mask)}
    if kind == "tune_all":
        planes = bcast + scat + scat + bool(mask & 0x2ED)  # Broadcast, Scatter, Gather, Reduce
        barrier = float(n_t) * n_P
        return {"bytes": table_in + 13.0 * (cells * planes + barrier), "flops": model_ops(mask) + model_ops(mask & SCATTER) + model_ops(mask & 0x2ED) + 8 * barrier}
    if kind == "study":
        surface = float(n_t) * len(_few_process_counts(case)) * n_m * len(s) * len(segs)
        return {"bytes": table_in + 8 * surface + cells * 24 * len(segs) + 4 * cells, "flops": 2 * surface + 3 * cells * len(segs)}
    return {"bytes": table_in + 13.0 * cells * (bcast + scat), "flops": model_ops(mask)}


def tolerance(case):
    # Times are IEEE doubles.  The only long sums are the Scatter Chain's: added one after another, the 65535 terms of the
    # longest case end within 7e-15 of the sum in extended precision (numpy on the CPU, this file's tables), 4e-16 in the
    # 2-norm; a closed form or another order is as good.  Everything else is a few roundings.  Picks may differ where two
    # times agree to the last bits, which one cell in a million may.
    return {"rel": 2e-15, "max": 3e-14, "differ": 1e-6}
