"""m = 3: groups of ranks are taken by pairs only where their pairs cost less
than the records they spare; with few first ranks of thousands of points each,
or few bits in the second rank, the groups are narrower or none.  Results are
those of the records (group_bits = 0)."""
import pytest

from gpu_helpers import torch
from paper_2305_16751_gb300 import domagg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,values0,values1,shared", [
    (300000, 200, 8, False),        # 3000 points a rank, S = 1: 6000 > 160 x 1 x 3
    (300000, 200, 1 << 24, False),  # 6000 > 160 x 1 x 20
    (100000, 200, 2, False),        # 2000 > 160
    (100000, 200, 1 << 24, True),   # 2000 <= 160 x 18
    (20000, 1 << 24, 2, True),      # narrower groups
    (20000, 1 << 24, 1 << 24, True)])
def test_groups_where_their_pairs_pay(n, values0, values1, shared):
    t = torch()
    g = t.Generator(device="cuda").manual_seed(10270)
    D, Q = (t.randint(0, 1 << 24, (n, 3), dtype=t.int32, device="cuda", generator=g) for _ in range(2))
    for x in (D, Q):
        x[:, 0] %= values0
        x[:, 1] %= values1
    w = t.randint(-1000, 1001, (n,), dtype=t.int64, device="cuda", generator=g)
    h = domagg.handle(0)
    domagg.domagg_set_tuning(h, "nodes", 0)
    try:
        out = domagg.forward(D, Q, w, "sum")
        assert (domagg.stats()["n_records_shared"] > 0) == shared
        domagg.domagg_set_tuning(h, "group_bits", 0)
        assert t.equal(out, domagg.forward(D, Q, w, "sum"))
    finally:
        domagg.domagg_set_tuning(h, "group_bits", 13)
        domagg.domagg_set_tuning(h, "nodes", 1)
    plan = domagg.BatchPlan([(D, Q, w)], "sum", headroom=0.1)
    try:
        plan.run()
        plan.status()
        assert t.equal(plan.outs[0], out)
    finally:
        plan.close()


def test_groups_stay_where_the_levels_above_go_by_items():
    """The empirical CDF at 2^20 points: 4600 points a group on average, more
    than the records of two levels would pay for, but a level less by items
    halves the nodes."""
    t = torch()
    g = t.Generator(device="cuda").manual_seed(10280)
    X = (t.randn((1 << 20, 3), device="cuda", generator=g) * 256).round() / 256
    h = domagg.handle(0)
    domagg.domagg_timing_read(h)
    domagg.domagg_timing_enable(h, True)
    try:
        out = domagg.forward(X, X, None, "count", nonstrict=7)
        kinds = domagg.domagg_timing_read(h)
    finally:
        domagg.domagg_timing_enable(h, False)
    # the items, from the algorithmic bytes of their two kernels (256 per
    # 32-point chunk, 12 + 20 per item): a level holds every point once, as
    # datum or as query; the two levels below the groups hold none
    items = (kinds["expand"]["bytes"] - 2**21 / 32 * 256) / 32
    assert 0 < items <= (domagg.stats()["rank_bits"][0] - 2) * 2**20, items / 2**20
    domagg.domagg_set_tuning(h, "nodes", 0)
    try:
        assert t.equal(out, domagg.forward(X, X, None, "count", nonstrict=7))
    finally:
        domagg.domagg_set_tuning(h, "nodes", 1)
