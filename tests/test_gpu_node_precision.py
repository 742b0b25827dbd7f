"""Float32 sums of m = 3 by nodes are as accurate as by records in HBM: a
node's answer joins the query's sum as a float-float pair, not rounded to one
float32 per level."""
import numpy as np
import pytest

from gpu_helpers import torch
from paper_2305_16751_gb300 import domagg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,signed", [(1 << 18, False), (1 << 18, True), (1 << 20, False)])
def test_nodes_are_as_accurate_as_records(n, signed):
    """Weights are multiples of 2^-20, so an int64 sum is exact; counted are
    the outputs that are not that sum rounded once.  By records, a query's
    part of a level is a float32 per second-rank record; by nodes only the
    nodes' deepest levels are (a part of the same sum), so the nodes' count
    is the smaller one; 2 % are left for chance."""
    t = torch()
    g = t.Generator(device="cuda").manual_seed(10400 + n % 7)
    D = t.rand((n, 3), device="cuda", generator=g)
    Q = t.rand((n, 3), device="cuda", generator=g)
    k = t.randint(-(1 << 24) if signed else 0, 1 << 24, (n,), device="cuda", generator=g)
    w = (k.double() * 2.0**-20).float()
    assert t.equal(w.double() * 2.0**20, k.double())
    exact = (domagg.forward(D, Q, k, "sum").double() * 2.0**-20).float()  # (below 2^53)
    h = domagg.handle(0)
    wrong = {}
    for nodes in (2, 0):
        domagg.domagg_set_tuning(h, "nodes", nodes)
        try:
            wrong[nodes] = int((domagg.forward(D, Q, w, "sum") != exact).sum())
        finally:
            domagg.domagg_set_tuning(h, "nodes", 1)
    print(n, signed, wrong)
    assert wrong[2] <= 1.02 * wrong[0], wrong
