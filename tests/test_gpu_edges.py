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
