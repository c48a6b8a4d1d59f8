"""GPU calls at the edges of what they accept."""
from dataclasses import replace

import numpy as np
import pytest

from paper_cs_0408034_b200 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def plogp():
    import torch
    assert torch.cuda.is_available()
    from paper_cs_0408034_b200 import plogp as mod
    return mod


@pytest.mark.parametrize("ids", [(9,), (2, 9), (5,), (2, 5, 9), range(13)])
@pytest.mark.parametrize("n_s", [1, 31, 32, 33, 64])
def test_lower_envelope_where_every_time_overflows(plogp, ids, n_s):
    """Gaps near the largest double: g(s) k and all times of the segmented strategies are infinite, for some message sizes
    with every candidate.  Both searches then choose the lowest id and the smallest size."""
    base = wl.config4(n_tables=2, P_hi=40, n_m=5, seed_offset=n_s)
    w = replace(base, m=np.array([4, 4096, 1 << 20, 1 << 24, 1 << 26], dtype=np.uint64), s_list=np.arange(4, 4 + 4 * n_s, 4, dtype=np.uint64),
                gaps=np.full_like(base.gaps, 1.5e308), strategy_mask=sum(1 << i for i in ids))
    with plogp.Tables.from_workload(w) as tabs:
        a, b = plogp.select_best(tabs, w), plogp.select_best(tabs, replace(w, search_mode=1))
        for x, y in ((a.strategy, b.strategy), (a.s_bytes, b.s_bytes), (a.time, b.time)):
            assert x[:, 0].equal(y[:, 0])
        assert 0 in ids or np.isposinf(a.time[:, 0, :, 1:].cpu().numpy()).all()


@pytest.mark.parametrize("scale", [1.0, 1e6, 1e8, 1e10, 1e12])
@pytest.mark.parametrize("n_s,n_P,listed,k_mode", [(64, 600, False, 0), (40, 2000, False, 1), (64, 30, True, 0), (70, 40, True, 1), (3000, 2000, False, 0), (3000, 2000, False, 1),
                                                   (9000, 300, False, 0), (20000, 60, True, 0), (9000, 9, True, 1)])
def test_lower_envelope_of_lines_that_differ_by_rounding(plogp, scale, n_s, n_P, listed, k_mode):
    """A latency far above the gaps makes the Segmented Chain's slopes equal but for a few last bits and many candidates' times
    equal after rounding: the smallest size among them is found as by the exhaustive search, bit for bit.  Short lists, long
    ones and one of several windows; process counts in a range, listed and listed far apart."""
    base = wl.config4(n_tables=12, P_hi=n_P + 1, n_m=3, seed_offset=n_s + n_P)
    w = replace(base, m=np.array([5000, 65536, 1000000, 1 << 24], dtype=np.uint64), s_list=None, s_lo=4, s_hi=4 * n_s, s_step=4, latency=base.latency * scale,
                strategy_mask=(1 << 5) | (1 << 3), k_mode=k_mode)
    if listed:
        w = replace(w, P_list=np.unique(np.rint(2 * 1e5 ** (np.arange(n_P) / (n_P - 1)))).astype(np.int32))
    with plogp.Tables.from_workload(w) as tabs:
        a, b = plogp.select_best(tabs, w), plogp.select_best(tabs, replace(w, search_mode=1))
        for x, y in ((a.strategy, b.strategy), (a.s_bytes, b.s_bytes), (a.time, b.time)):
            assert x[:, 0].equal(y[:, 0])
        a, b = plogp.predict(tabs, w), plogp.predict(tabs, replace(w, search_mode=1))
        assert a.time[:, 5].equal(b.time[:, 5]) and a.best_s[:, 1].equal(b.best_s[:, 1])


def off_by_one(x):
    """A tensor like x (its contents too) one element behind the start of an allocation."""
    import torch
    y = torch.empty(x.numel() + 1, dtype=x.dtype, device=x.device)[1:].view(x.shape)
    y.copy_(x)
    return y


@pytest.mark.parametrize("n_tables,n_m,n_P,n_s,listed", [(1, 20, 40, 7, False), (4, 64, 600, 33, True), (600, 64, 24, 9, False), (40, 128, 512, 20, False), (11500, 46, 16, 3, False),
                                                         (120, 130, 560, 5, False)])
def test_outputs_at_odd_addresses(plogp, n_tables, n_m, n_P, n_s, listed):
    """Outputs and inputs aligned for single elements only: the stores of two and four cells give way to single ones on grids
    that take them otherwise (even n_m, rows off the sectors, sensitivity planes, boundaries of 8 and 16 bytes), with the
    same decisions and times (Scatter Chain sums to 1e-12: another order of additions)."""
    import torch
    w = wl.config4(n_tables=n_tables, P_hi=n_P + 1, n_m=n_m, n_s=n_s, seed_offset=n_P)
    if listed:
        w = replace(w, P_list=(2 + 3 * np.arange(n_P)).astype(np.int32))
    with plogp.Tables.from_workload(w) as tabs:
        dec, pred = plogp.select_best(tabs, w), plogp.predict(tabs, w)
        d = plogp.DecisionTable(*(off_by_one(torch.zeros_like(x)) for x in (dec.strategy, dec.s_bytes, dec.time)))
        plogp.select_best(tabs, w, out=d)
        assert d.strategy.equal(dec.strategy) and d.s_bytes.equal(dec.s_bytes)
        assert d.time[:, 0].equal(dec.time[:, 0]) and torch.allclose(d.time[:, 1], dec.time[:, 1], rtol=1e-12, atol=0.0)
        p = plogp.Prediction(off_by_one(torch.zeros_like(pred.time)), off_by_one(torch.zeros_like(pred.best_s)))
        plogp.predict(tabs, w, out=p)
        assert p.best_s.equal(pred.best_s) and p.time[:, :11].equal(pred.time[:, :11]) and p.time[:, 12].equal(pred.time[:, 12])
        assert torch.allclose(p.time[:, 11], pred.time[:, 11], rtol=1e-12, atol=0.0)
        (fixed, ratio), (f2, r2) = (plogp.segment_sensitivity(tabs, w, 8192, pred=x) for x in (pred, plogp.Prediction(off_by_one(pred.time), None)))
        assert f2.equal(fixed) and r2.equal(ratio)
        a, b = plogp.decision_boundaries(dec), plogp.decision_boundaries(plogp.DecisionTable(off_by_one(dec.strategy), None, None))
        assert a.equal(b)
