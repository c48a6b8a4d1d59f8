"""GPU parity where the FP32 lower bounds of the segment search decide what is looked at in FP64: tilings of the process
counts and candidates at their edges, and tables whose times lie far outside FP32's range."""
from dataclasses import replace

import numpy as np
import pytest

from paper_cs_0408034_b200 import workloads as wl
from parity import check_decision, check_prediction, oracle_tables

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def plogp():
    import torch
    assert torch.cuda.is_available()
    from paper_cs_0408034_b200 import plogp as mod
    return mod


def both(plogp, w):
    """Decision table and predictions of every cell against the oracle (times to 1e-12, picks exact: tests/parity.py)."""
    import torch
    ot = oracle_tables(w)
    with plogp.Tables.from_workload(w) as tabs:
        dec = plogp.select_best(tabs, w)
        pred = plogp.predict(tabs, w)
        torch.cuda.synchronize()
        assert check_decision(w, ot, dec) + check_prediction(w, ot, pred) > 0


@pytest.mark.parametrize("n_P,ids,k_mode", [(1, (2, 5, 9), 0), (31, (5,), 1), (256, (2, 5), 0), (257, (9,), 0), (700, (2, 9), 1),
                                            (1100, (2, 5, 9), 0), (2049, (0, 2, 5, 7), 0)])
def test_long_lists_at_the_edges_of_the_process_count_tiles(plogp, n_P, ids, k_mode):
    """1, 2, 4 and 8 tiles of 256 process counts per CTA (the warps then split the candidates 8, 4, 2 and 1 ways), and a
    candidate list that ends inside a sub-chunk of 256."""
    base = wl.config4(n_tables=2, P_hi=n_P + 1, n_m=5, seed_offset=70 + n_P)
    both(plogp, replace(base, s_list=None, s_lo=4, s_hi=4 * 700, s_step=4, strategy_mask=sum(1 << i for i in ids), k_mode=k_mode))


def test_long_list_over_several_chunks(plogp):
    """A list of 2300 sizes: two chunks of candidates per message size, the optimum in either."""
    base = wl.config4(n_tables=2, P_hi=90, n_m=4, seed_offset=5)
    both(plogp, replace(base, m=np.array([4, 3000, 9000, 400000], dtype=np.uint64), s_list=None, s_lo=4, s_hi=9200, s_step=4))


@pytest.mark.parametrize("scale", [1e-60, 1e-42, 1e36, 1e60])
@pytest.mark.parametrize("long_list", [False, True])
def test_times_outside_the_range_of_fp32(plogp, scale, long_list):
    """Below FP32's smallest number every bound is 0, above its largest every upper bound is infinite: all cells are
    then compared in FP64, and the results are the oracle's."""
    base = wl.config4(n_tables=2, P_hi=300, n_m=6, n_s=24, seed_offset=8)
    w = replace(base, gaps=base.gaps * scale, latency=base.latency * scale)
    if long_list:
        w = replace(w, P_hi=70, s_list=None, s_lo=4, s_hi=4 * 300, s_step=4)
    both(plogp, w)


@pytest.mark.parametrize("s_lo,s_step,n_s,k_mode", [(4, 4, 66, 0), (4, 4, 3000, 1), (4, 12, 900, 0), (1000, 20, 1500, 1), (20000, 4, 500, 0),
                                                    (4, 4000, 300, 0), (4, 4000, 300, 1)])
def test_envelope_over_equally_spaced_candidates(plogp, s_lo, s_step, n_s, k_mode):
    """The first candidate of every segment count, where counts change with every candidate, with some and with few of
    them, and where counts are skipped; message sizes below, inside and above the list."""
    base = wl.config4(n_tables=2, P_hi=130, n_m=4, seed_offset=n_s)
    m = np.array([4, 48, 1000, 3996, 4000, 4004, 20004, 65536, 1000000, 1 << 24], dtype=np.uint64)
    both(plogp, replace(base, m=m, s_list=None, s_lo=s_lo, s_hi=s_lo + s_step * (n_s - 1), s_step=s_step, k_mode=k_mode, search_mode=1))


def test_alternating_grids_keep_their_plans(plogp):
    """Twelve grids in turn on one handle (more than it keeps plans for), twice: every result is the one of a handle that
    has seen no other grid."""
    import torch
    base = wl.config4(n_tables=3, P_hi=40, n_m=9, n_s=12, seed_offset=3)
    grids = [replace(base, P_hi=10 + 3 * i, strategy_mask=wl.ALL_STRATEGIES if i % 3 else 0x1C07) for i in range(12)]
    fresh = []
    for w in grids:
        with plogp.Tables.from_workload(w) as tabs:
            fresh.append(plogp.select_best(tabs, w))
    with plogp.Tables.from_workload(base) as tabs:
        for w, f in list(zip(grids, fresh)) * 2:
            d = plogp.select_best(tabs, w)
            assert torch.equal(d.strategy, f.strategy) and torch.equal(d.s_bytes, f.s_bytes) and torch.equal(d.time, f.time)
        torch.cuda.synchronize()


@pytest.mark.parametrize("n_m", [7, 8, 16, 24, 32, 40])
@pytest.mark.parametrize("n_P", [1, 7, 8, 9, 17])
def test_boundaries_of_random_maps(plogp, n_m, n_P):
    """One byte, 8 and 16 bytes per thread; runs of 8 process counts that end inside, at and past a table's last row."""
    import torch
    from oracle import plogp_oracle as po
    rng = np.random.default_rng(n_m * 100 + n_P)
    s = rng.integers(0, 3, size=(3, 2, n_P, n_m)).astype(np.uint8) * 200  # neighbouring bytes must not touch one another
    dec = plogp.DecisionTable(torch.as_tensor(s, device="cuda"), None, None)
    assert np.array_equal(plogp.decision_boundaries(dec).cpu().numpy(), po.decision_boundaries(s))


@pytest.mark.parametrize("n_P,n_m,n_s,n_tables,listed,search", [(1, 1, 1, 1, False, 0), (3, 5, 64, 1, False, 0), (129, 33, 7, 1, True, 0), (257, 37, 33, 2, False, 1),
                                                               (600, 70, 20, 1, False, 0), (127, 300, 12, 1, True, 1), (1500, 64, 3, 2, False, 0)])
def test_both_halves_in_one_launch_and_in_two(plogp, n_P, n_m, n_s, n_tables, listed, search):
    """Small grids: one launch for both halves (tiles of 128 process counts, four warps per Scatter CTA); the same call
    with per-kernel timing on makes the two launches.  Both match the oracle and one another bit for bit."""
    import torch
    w = wl.config4(n_tables=n_tables, P_hi=n_P + 1, n_m=n_m, n_s=n_s, seed_offset=n_P)
    if listed:
        w = replace(w, P_list=np.unique(np.rint(2 * 1500 ** (np.arange(n_P) / max(1, n_P - 1)))).astype(np.int32))
    w = replace(w, search_mode=search)
    both(plogp, w)
    with plogp.Tables.from_workload(w) as tabs:
        a = plogp.select_best(tabs, w)
        plogp.profile_enable(tabs)
        b = plogp.select_best(tabs, w)
        torch.cuda.synchronize()
        assert len(plogp.profile_read(tabs)) >= 2
        assert torch.equal(a.strategy, b.strategy) and torch.equal(a.s_bytes, b.s_bytes) and torch.equal(a.time, b.time)


@pytest.mark.parametrize("n_m,n_P,n_s,k_mode", [(17, 300, 33, 0), (33, 257, 5, 1), (65, 129, 64, 0), (97, 513, 20, 0), (98, 70, 32, 0)])
def test_prediction_rows_off_the_sectors_on_many_tables(plogp, n_m, n_P, n_s, k_mode):
    """Rows of message sizes that are no multiple of 32 bytes, on enough tables for CTAs of 32 message sizes (the last one
    ragged): the first and last table match the oracle, and the searches of five tables at either end a call
    over these alone, bit for bit."""
    import torch
    n = 2368 // max(1, n_m // 16) + 8
    w = replace(wl.config4(n_tables=n, P_hi=n_P + 1, n_m=n_m, n_s=n_s, seed_offset=n_m), k_mode=k_mode)
    with plogp.Tables.from_workload(w) as tabs:
        a = plogp.predict(tabs, w)
    p_idx = np.unique(np.r_[0:n_P:7, n_P - 1])
    assert check_prediction(w, oracle_tables(w), a, tables=(0, n - 1), p_idx=p_idx) > 0
    for lo in (0, n - 5):
        few = replace(w, gaps=np.ascontiguousarray(w.gaps[lo:lo + 5]), latency=w.latency[lo:lo + 5])
        with plogp.Tables.from_workload(few) as tabs:
            b = plogp.predict(tabs, few)
        assert torch.equal(a.time[lo:lo + 5, [2, 5, 9]], b.time[:, [2, 5, 9]]) and torch.equal(a.best_s[lo:lo + 5], b.best_s)


@pytest.mark.parametrize("n_m,n_P,n_tables,listed,ids", [(33, 160, 796, False, range(13)), (35, 163, 736, True, (0, 1, 3, 10)), (255, 161, 103, False, (4, 6, 7, 8)),
                                                         (257, 409, 40, False, range(13)), (1031, 4100, 1, True, (0, 2, 6, 10, 11))])
def test_closed_form_planes_cell_by_cell(plogp, n_m, n_P, n_tables, listed, ids):
    """Planes written as they lie in memory (rows off the sectors, at least 2^22 cells): starts of planes at all 32 offsets
    from a 256-byte boundary, rows shorter and longer than a CTA, with and without the kernel of the Scatter sums behind."""
    base = wl.config4(n_tables=n_tables, P_hi=n_P + 1, n_m=n_m, n_s=3, seed_offset=n_P)
    w = replace(base, m=np.arange(4, 4 + 4 * n_m, 4, dtype=np.uint64) ** 2 // 4, strategy_mask=sum(1 << i for i in ids))
    if listed:
        w = replace(w, P_list=(2 + 3 * np.arange(n_P)).astype(np.int32))
    assert w.n_m == n_m and w.n_P == n_P and n_P * n_m * n_tables >= 1 << 22
    with plogp.Tables.from_workload(w) as tabs:
        pred = plogp.predict(tabs, w)
    p_idx, m_idx = np.unique(np.r_[0:4, 0:n_P:29, n_P - 2, n_P - 1]), np.unique(np.r_[0:n_m:7, n_m - 1])
    assert check_prediction(w, oracle_tables(w), pred, tables=sorted({0, n_tables // 2, n_tables - 1}), p_idx=p_idx, m_idx=m_idx) > 0


@pytest.mark.parametrize("n_m,n_P,n_tables,n_bp,listed,ids", [(45, 257, 740, 64, False, range(13)), (255, 161, 206, 12, True, range(13)), (97, 2000, 45, 256, False, (2, 10, 12)),
                                                              (150, 300, 200, 30, False, (5, 11)), (46, 16, 11500, 5, False, (10, 11, 12)), (129, 65100, 1, 100, True, (0, 11, 12))])
def test_scatter_rows_off_the_sectors(plogp, n_m, n_P, n_tables, n_bp, listed, ids):
    """Pieces of the Scatter plane per CTA (rows off the sectors, at least 2^23 cells): ragged last runs and flushes, pieces
    that start at all four offsets from a group of cells, one to eight warps, sums in front of a run, some ids alone."""
    base = wl.config4(n_tables=n_tables, P_hi=n_P + 1, n_m=n_m, n_s=3, seed_offset=n_P)
    sizes = wl.log_spaced_multiples(4, 256 << 20, n_bp)
    gaps = np.stack([np.interp(sizes.astype(float), base.sizes.astype(float), g) for g in base.gaps])
    w = replace(base, sizes=sizes, gaps=gaps, strategy_mask=sum(1 << i for i in ids))
    if listed:
        w = replace(w, P_list=(2 + 2 * np.arange(n_P)).astype(np.int32))
    assert w.n_P == n_P and n_P * n_m * n_tables >= 1 << 23
    p_idx, m_idx = np.unique(np.r_[0:4, 0:n_P:max(1, n_P // 40), n_P - 2, n_P - 1]), np.unique(np.r_[0:n_m:11, n_m - 1])
    ot = oracle_tables(w)
    sample = dict(tables=sorted({0, 1 % n_tables, n_tables // 2, n_tables - 1}), p_idx=p_idx, m_idx=m_idx)
    with plogp.Tables.from_workload(w) as tabs:
        assert check_decision(w, ot, plogp.select_best(tabs, w), **sample) > 0
        assert check_prediction(w, ot, plogp.predict(tabs, w), **sample) > 0


@pytest.mark.parametrize("n_bp,n_P,n_m,first,ids", [(2, 1, 33, 2, (10, 11, 12)), (3, 40, 5, 900, (11,)), (9, 33, 64, 2, (11, 12)), (96, 301, 97, 3, range(13)), (97, 301, 97, 3, range(13))])
def test_listed_scatter_sums_by_interval(plogp, n_bp, n_P, n_m, first, ids):
    """Sums per table interval for listed process counts: fewer intervals than warps, lists that start far from 2 and skip
    intervals, arguments below and above the table, message sizes with idle lanes, the longest table that takes them."""
    n = 1400 // n_m + 8
    base = wl.config4(n_tables=n, P_hi=5000, n_m=n_m, n_s=3, seed_offset=n_bp)
    sizes = wl.log_spaced_multiples(64, 64 << 20, n_bp)
    gaps = np.stack([np.interp(sizes.astype(float), base.sizes.astype(float), g) for g in base.gaps])
    P_list = np.unique(np.r_[first, first + np.rint(1.03 ** np.arange(n_P * 3)).astype(int)])[:n_P].astype(np.int32)
    w = replace(base, sizes=sizes, gaps=gaps, strategy_mask=sum(1 << i for i in ids), P_list=P_list)
    ot = oracle_tables(w)
    with plogp.Tables.from_workload(w) as tabs:
        plogp.profile_enable(tabs)  # two launches
        assert check_decision(w, ot, plogp.select_best(tabs, w), tables=(0, 1, n - 1)) > 0


@pytest.mark.parametrize("n_m,n_P,n_s,search", [(16, 257, 32, 0), (17, 300, 32, 1), (40, 250, 8, 0), (64, 520, 33, 0), (33, 700, 20, 1), (41, 512, 64, 0), (24, 512, 57, 1)])
def test_decisions_on_many_tables(plogp, n_m, n_P, n_s, search):
    """Grids of many CTAs (five per SM where their shared memory fits): the first and last table match the oracle, five
    tables at either end a call over these alone (fewer CTAs per SM, other tiles), bit for bit in the Broadcast half."""
    import torch
    n = 2368 // max(1, n_m // 16) + 8
    w = replace(wl.config4(n_tables=n, P_hi=n_P + 1, n_m=n_m, n_s=n_s, seed_offset=n_m), search_mode=search)
    with plogp.Tables.from_workload(w) as tabs:
        a = plogp.select_best(tabs, w)
    assert check_decision(w, oracle_tables(w), a, tables=(0, n - 1), p_idx=np.unique(np.r_[0:n_P:7, n_P - 1])) > 0
    for lo in (0, n - 5):
        few = replace(w, gaps=np.ascontiguousarray(w.gaps[lo:lo + 5]), latency=w.latency[lo:lo + 5])
        with plogp.Tables.from_workload(few) as tabs:
            b = plogp.select_best(tabs, few)
        for x, y in ((a.strategy, b.strategy), (a.s_bytes, b.s_bytes), (a.time, b.time)):
            assert torch.equal(x[lo:lo + 5, 0], y[:, 0])


@pytest.mark.parametrize("n_tables,n_m,n_P,search", [(100, 33, 512, 0), (110, 56, 300, 1), (40, 129, 700, 0)])
def test_decisions_on_a_few_ctas_per_sm(plogp, n_tables, n_m, n_P, search):
    """Grids of a few CTAs per SM, the last group of message sizes ragged."""
    w = replace(wl.config4(n_tables=n_tables, P_hi=n_P + 1, n_m=n_m, n_s=24, seed_offset=n_m), search_mode=search)
    with plogp.Tables.from_workload(w) as tabs:
        a, b = plogp.select_best(tabs, w), plogp.predict(tabs, w)
    ot, sample = oracle_tables(w), dict(tables=(0, n_tables - 1), p_idx=np.unique(np.r_[0:n_P:5, n_P - 1]))
    assert check_decision(w, ot, a, **sample) + check_prediction(w, ot, b, **sample) > 0
