"""GPU parity of the Broadcast half and the segmented planes on short candidate lists: lines ruled out for ranges of process
counts, message sizes side by side in 8, 16 or 32 threads or all of a table's in a CTA."""
from dataclasses import replace

import numpy as np
import pytest

from oracle import plogp_oracle as po
from paper_cs_0408034_b200 import workloads as wl
from parity import check_decision, check_prediction, oracle_sgrid, oracle_tables

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def plogp():
    import torch
    assert torch.cuda.is_available()
    from paper_cs_0408034_b200 import plogp as mod
    return mod


def both(plogp, w, tables=None):
    """Decision table and predictions against the oracle (times to 1e-12, picks exact: tests/parity.py)."""
    import torch
    ot = oracle_tables(w)
    with plogp.Tables.from_workload(w) as tabs:
        dec = plogp.select_best(tabs, w)
        pred = plogp.predict(tabs, w)
        torch.cuda.synchronize()
        assert check_decision(w, ot, dec, tables=tables) + check_prediction(w, ot, pred, tables=tables) > 0


@pytest.mark.parametrize("n_m", [1, 8, 9, 16, 17, 32, 33])
@pytest.mark.parametrize("n_s,n_P,k_mode", [(1, 1, 0), (31, 7, 1), (32, 65, 0), (33, 130, 0), (64, 513, 1)])
def test_widths_and_steps(plogp, n_m, n_s, n_P, k_mode):
    both(plogp, wl_grid(n_tables=2, n_P=n_P, n_m=n_m, n_s=n_s, k_mode=k_mode))


def wl_grid(n_tables, n_P, n_m, n_s, k_mode=0, P_lo=2):
    w = wl.config4(n_tables=n_tables, P_hi=P_lo + n_P - 1, n_m=n_m, n_s=n_s, seed_offset=n_P + n_m)
    return replace(w, P_lo=P_lo, k_mode=k_mode)


@pytest.mark.parametrize("ids", [(0,), (1, 2), (2,), (3, 5), (4, 5), (5,), (9,), (2, 9), (1, 4, 8), (0, 3, 6), (2, 5, 7), range(10)])
def test_strategies_alone_and_together(plogp, ids):
    """Lines without pairs, pairs without lines, rendezvous variants with and without their siblings, whole messages."""
    w = wl_grid(n_tables=2, n_P=90, n_m=20, n_s=20)
    m = np.unique(np.concatenate([w.m, w.s_list[3:6]]))  # a candidate of the whole message's size
    both(plogp, replace(w, m=m, s_list=w.s_list[2:], strategy_mask=sum(1 << i for i in ids)))


@pytest.mark.parametrize("kind", ["flat", "stairs", "falls", "latency"])
@pytest.mark.parametrize("n_s", [20, 64])
def test_lines_close_to_one_another(plogp, kind, n_s):
    """Equal gaps over many sizes, gaps that fall, a latency far above the gaps: many candidates within rounding."""
    w = wl_grid(n_tables=3, n_P=300, n_m=12, n_s=n_s)
    g = w.gaps.copy()
    if kind == "flat":
        g[:, :] = g[:, :1]
    elif kind == "stairs":
        g = np.repeat(g[:, ::8], 8, axis=1)
    elif kind == "falls":
        g[:, 5:40:3] *= 0.5
    both(plogp, replace(w, gaps=np.ascontiguousarray(g), latency=w.latency * (1e9 if kind == "latency" else 1.0)))


@pytest.mark.parametrize("n_m,n_P,n_s,listed,n_tables", [
    (17, 21, 9, False, 300), (33, 520, 33, False, 300), (50, 16, 8, False, 300), (127, 40, 20, True, 300), (129, 9, 64, False, 300), (255, 33, 5, False, 300), (256, 8, 3, False, 300),
    (33, 97, 33, False, 900), (33, 511, 24, True, 900), (127, 257, 24, False, 900), (201, 256, 3, True, 900), (173, 300, 1, False, 900), (99, 520, 9, False, 450),
    (145, 31, 9, False, 900), (65, 14, 40, True, 900), (195, 172, 8, False, 900), (35, 1100, 32, False, 300), (34, 193, 20, False, 600), (52, 257, 32, False, 600), (250, 260, 32, True, 600), (255, 256, 20, False, 600)])
def test_all_message_sizes_in_a_cta(plogp, n_m, n_P, n_s, listed, n_tables):
    """Many tables, rows off the sectors: the cells of a step put together in shared memory, for the predictions and the decision
    (600 tables: the predictions alone; 300 of few process counts: neither).  The same as with outputs aligned for single
    elements, which are stored one by one, and as the oracle's for some tables."""
    import torch
    w = wl_grid(n_tables=n_tables, n_P=n_P, n_m=n_m, n_s=n_s)
    if listed:
        w = replace(w, P_list=(2 + 3 * np.arange(n_P)).astype(np.int32))
    both(plogp, w, tables=[0, n_tables // 2 + 1, n_tables - 1])

    def off_by_one(x):
        return torch.zeros(x.numel() + 1, dtype=x.dtype, device=x.device)[1:].view(x.shape)

    with plogp.Tables.from_workload(w) as tabs:
        dec, pred = plogp.select_best(tabs, w), plogp.predict(tabs, w)
        d = plogp.DecisionTable(*(off_by_one(x) for x in (dec.strategy, dec.s_bytes, dec.time)))
        plogp.select_best(tabs, w, out=d)
        p = plogp.Prediction(off_by_one(pred.time), off_by_one(pred.best_s))
        plogp.predict(tabs, w, out=p)
        for a, b in ((d.strategy, dec.strategy), (d.s_bytes, dec.s_bytes), (d.time, dec.time)):
            assert a[:, 0].equal(b[:, 0])
        assert p.best_s.equal(pred.best_s) and all(p.time[:, i].equal(pred.time[:, i]) for i in (2, 5, 9))


@pytest.mark.parametrize("n_m,n_s,octaves", [(255, 64, 0), (253, 24, 0), (201, 32, 0), (250, 32, 0), (229, 8, 29), (255, 24, 29), (255, 32, 29), (157, 20, 29)])
def test_more_than_a_cta_has_room_for(plogp, n_m, n_s, octaves):
    """Many tables, rows off the sectors, long lists and process counts over many (floor, ceil) pairs of log2 P: all message sizes
    together would take more shared memory than a CTA, or than half of an SM, has."""
    w = wl_grid(n_tables=900, n_P=300, n_m=n_m, n_s=n_s)
    if octaves:  # P m < 2^53; the oracle would add up the Scatter Chain's terms one by one
        P = np.unique(np.concatenate([1 << np.arange(1, octaves), np.rint(2.0 ** np.linspace(1.5, octaves - 0.5, 256))]))
        w = replace(w, P_list=P.astype(np.int32), m=256 * np.arange(1, n_m + 1, dtype=np.uint64), strategy_mask=0x17FF)
    both(plogp, w, tables=[0, 899])


@pytest.mark.parametrize("kind", ["as drawn", "flat", "stairs", "falls"])
@pytest.mark.parametrize("n_s,s_step,n_P,k_mode", [(255, 4, 40, 0), (257, 8, 256, 1), (2600, 4, 257, 0), (700, 400, 530, 0)])
def test_long_lists_bounded_by_their_ends(plogp, kind, n_s, s_step, n_P, k_mode):
    """Sub-chunks of 256 candidates passed over by the smallest gap between their first and last size: breakpoints inside one,
    several sub-chunks between two breakpoints, gaps that fall; process counts in the first 256 and behind them."""
    w = wl_grid(n_tables=2, n_P=n_P, n_m=4, n_s=1, k_mode=k_mode)
    g = w.gaps.copy()
    if kind == "flat":
        g[:, :] = g[:, :1]
    elif kind == "stairs":
        g = np.repeat(g[:, ::8], 8, axis=1)
    elif kind == "falls":
        g[:, 3:60:4] *= 0.3
    both(plogp, replace(w, gaps=np.ascontiguousarray(g), m=np.array([500, 30000, 1 << 20, 1 << 24], dtype=np.uint64), s_list=None, s_lo=4, s_hi=4 + s_step * (n_s - 1),
                        s_step=s_step, strategy_mask=0x224))


def picks_as_the_oracle(plogp, w, tables):
    """Strategies and segment sizes of Broadcast equal to the oracle's everywhere, on ties too, and times bit for bit."""
    import torch
    ot, sg = oracle_tables(w), oracle_sgrid(w)
    with plogp.Tables.from_workload(w) as tabs:
        dec, pred = plogp.select_best(tabs, w), plogp.predict(tabs, w)
        torch.cuda.synchronize()
    for t in tables:
        o = po.predict_grid(ot[t], w.strategy_mask, w.P_values(), w.m, sg, w.k_mode)
        d = po.select_grid(w.strategy_mask, o)
        np.testing.assert_array_equal(dec.strategy[t, 0].cpu().numpy(), d.strategy[0])
        np.testing.assert_array_equal(dec.s_bytes[t, 0].cpu().numpy().view(np.uint32), d.s[0])
        np.testing.assert_array_equal(dec.time[t, 0].cpu().numpy(), d.time[0])
        for q, sid in enumerate(po.SEGMENTED_IDS):
            if (w.strategy_mask >> sid) & 1:
                np.testing.assert_array_equal(pred.best_s[t, q].cpu().numpy().view(np.uint32), o.best_s[q])
                np.testing.assert_array_equal(pred.time[t, sid].cpu().numpy(), o.time[sid])


@pytest.mark.parametrize("ids", [range(10), (2, 5, 9), (4, 5), (1, 2, 4, 5, 8, 9), (0, 2), (3, 5), (8, 9), (1, 2, 5)])
@pytest.mark.parametrize("n_tables,n_m,n_P,k_mode", [(40, 19, 70, 0), (300, 33, 70, 1)])
def test_ties_go_to_the_lowest_id_and_size(plogp, ids, n_tables, n_m, n_P, k_mode):
    """Whole gaps at powers of two: every product and sum of the models is exact, however it is rounded on the way, and many
    are equal."""
    rng = np.random.default_rng(n_m)
    gaps = np.cumsum(rng.integers(0, 2, (n_tables, 21)) * rng.integers(0, 2, (n_tables, 1)), axis=1).astype(np.float64)
    w = replace(wl_grid(n_tables=n_tables, n_P=n_P, n_m=n_m, n_s=8, k_mode=k_mode), sizes=(1 << np.arange(21)).astype(np.uint64), gaps=gaps,
                latency=rng.integers(0, 3, n_tables).astype(np.float64), strategy_mask=sum(1 << i for i in ids),
                s_list=np.array([64, 128, 192, 256, 1024, 4096, 4100, 65536], dtype=np.uint64))
    m = np.unique(np.concatenate([w.s_list, [4, 16, 8192, 1 << 20], np.arange(1, n_m) * 516]).astype(np.uint64))[:n_m]
    picks_as_the_oracle(plogp, replace(w, m=m), range(0, n_tables, 7))


def test_rendezvous_times_that_round_to_the_others(plogp):
    """Handshakes of less than a rounding of the gap: where no candidate fits, ids 4 and 5 cost the same at some process counts
    and differ by their last bit at others."""
    rng = np.random.default_rng(4)
    c = 1.0 + rng.random(64)
    gaps = np.stack([np.zeros(64), c, c, c], axis=1)
    w = replace(wl_grid(n_tables=64, n_P=63, n_m=1, n_s=1), sizes=np.array([1, 1024, 1 << 20, 1 << 21], dtype=np.uint64), gaps=gaps,
                latency=np.where(np.arange(64) < 60, rng.uniform(0.34, 0.49, 64) * 2.0**-52, 1e-25), s_list=np.array([1 << 16, 1 << 18], dtype=np.uint64),
                m=np.array([1024, 4096, 32768], dtype=np.uint64), strategy_mask=0x30)
    picks_as_the_oracle(plogp, w, range(64))


@pytest.mark.parametrize("n_s", [(1 << 31) - 1, (1 << 31) - 200, (1 << 31) - (1 << 20) - 1])
def test_candidate_indices_up_to_the_last(plogp, n_s):
    """Every size up to n_s is a candidate and the gap is the same for all: fewer segments are better, and the best size is the
    message's own, the last candidate for the longest message."""
    import torch
    m = np.array([4096, 1 << 30, n_s], dtype=np.uint64)
    grid = plogp.GridArgs(m, np.array([2, 3, 40, 300], dtype=np.int32), 2, 2, None, s_lo=1, s_hi=n_s, s_step=1, dtype_bytes=1, strategy_mask=0x224)
    with plogp.Tables(np.array([1, 1 << 20], dtype=np.uint64), np.array([[3.0, 3.0]]), np.array([0.5])) as tabs:
        dec, pred = plogp.select_best(tabs, grid), plogp.predict(tabs, grid)
        torch.cuda.synchronize()
    for x in (dec.s_bytes[0, 0], *pred.best_s[0]):
        np.testing.assert_array_equal(x.cpu().numpy().view(np.uint32), np.broadcast_to(m, (4, 3)))
    # the Segmented Binomial Tree of one segment: floor(log2 P) 3 + ceil(log2 P) 0.5
    np.testing.assert_array_equal(dec.time[0, 0].cpu().numpy(), np.broadcast_to([[3.5], [4.0], [18.0], [28.5]], (4, 3)))


@pytest.mark.parametrize("n_P,n_m,n_s,k_mode,listed,ids", [
    (1, 1, 1, 0, False, range(13)), (127, 1, 3, 1, False, range(13)), (16, 8, 64, 0, False, range(13)), (43, 3, 33, 0, True, range(13)), (70, 19, 8, 1, False, range(10)),
    (70, 19, 8, 0, True, (2, 9)), (30, 33, 20, 0, False, (0, 3, 5, 6, 7, 10, 11, 12)), (20, 40, 16, 1, False, (1, 4, 5, 8)), (9, 7, 64, 0, False, (5,)), (64, 2, 12, 0, False, (1, 2, 9, 12))])
def test_a_cell_per_thread_as_lines(plogp, n_P, n_m, n_s, k_mode, listed, ids):
    """The same tables once and 300 times: small grids have a cell per thread, large ones lines for ranges of process counts.
    Times and picks are the same, bit for bit, and the oracle's."""
    import torch
    w = wl_grid(n_tables=3, n_P=n_P, n_m=n_m, n_s=n_s, k_mode=k_mode, P_lo=3 if k_mode else 2)
    if listed:
        w = replace(w, P_list=(2 + 5 * np.arange(n_P)).astype(np.int32))
    w = replace(w, strategy_mask=sum(1 << i for i in ids), m=np.unique(np.concatenate([w.m[: max(1, n_m - 2)], w.s_list[-1:]])))
    both(plogp, w)
    many = replace(w, gaps=np.tile(w.gaps, (300, 1)), latency=np.tile(w.latency, 300))
    with plogp.Tables.from_workload(w) as a, plogp.Tables.from_workload(many) as b:
        x, y = plogp.select_best(a, w), plogp.select_best(b, w)
        p, q = plogp.predict(a, w), plogp.predict(b, w)
        r, s = plogp.select_best_collective(a, w, plogp.REDUCE), plogp.select_best_collective(b, w, plogp.REDUCE)
        torch.cuda.synchronize()
    for first in (0, 3 * 299):
        for u, v in ((x.strategy, y.strategy), (x.s_bytes, y.s_bytes), (x.time, y.time)):
            assert u[:, 0].equal(v[first:first + 3, 0])
        for u, v in ((r.strategy, s.strategy), (r.s_bytes, s.s_bytes), (r.time, s.time)):
            assert u.equal(v[first:first + 3])
        for j, i in enumerate(po.SEGMENTED_IDS):
            if i in ids:
                assert p.time[:, i].equal(q.time[first:first + 3, i]) and p.best_s[:, j].equal(q.best_s[first:first + 3, j])


@pytest.mark.parametrize("n_tables,n_P,n_m,n_s", [(72, 200, 25, 4), (72, 713, 25, 8), (200, 99, 9, 10), (16, 600, 64, 32), (64, 511, 37, 16), (48, 1384, 24, 10), (4, 2696, 33, 14)])
def test_tilings_of_medium_grids(plogp, n_tables, n_P, n_m, n_s):
    """Fewer and larger CTAs: both halves in one launch, predictions of few candidates."""
    both(plogp, wl_grid(n_tables=n_tables, n_P=n_P, n_m=n_m, n_s=n_s), tables=[0, n_tables - 1])


@pytest.mark.parametrize("ids", [(2, 5), (9,), (2, 5, 9), range(10)])
@pytest.mark.parametrize("n_s,s_step,k_mode,P_lo", [(65, 4, 0, 2), (600, 4, 1, 2), (3000, 64, 0, 250), (2049, 4, 0, 2)])
def test_ties_in_long_lists(plogp, ids, n_s, s_step, k_mode, P_lo):
    """Whole gaps at powers of two, equal over many of them, and long lists of candidates: exact products, many equal times.
    Sub-chunks and groups that are passed over hold none that is better, nor a smaller size as good."""
    rng = np.random.default_rng(n_s)
    gaps = np.cumsum(rng.integers(0, 2, (8, 21)) * rng.integers(0, 2, (8, 21)) * rng.integers(0, 2, (8, 1)), axis=1).astype(np.float64) + 1.0
    w = replace(wl_grid(n_tables=8, n_P=280, n_m=1, n_s=1, k_mode=k_mode, P_lo=P_lo), sizes=(1 << np.arange(21)).astype(np.uint64), gaps=gaps,
                latency=rng.integers(0, 3, 8).astype(np.float64), strategy_mask=sum(1 << i for i in ids), s_list=None, s_lo=4, s_hi=4 + s_step * (n_s - 1), s_step=s_step,
                m=np.array([4, 512, 1024, 6000, 65536, 100000, 1 << 20], dtype=np.uint64))
    picks_as_the_oracle(plogp, w, range(8))
