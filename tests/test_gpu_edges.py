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
