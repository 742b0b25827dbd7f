"""m = 3 calls of 2^19 points and more take the nodes' path only where it
gains: with few distinct values in a coordinate a record costs no more than an
item, and the levels stay records in HBM; results either way are those of the
other path."""
import numpy as np
import pytest

import oracle
from gpu_helpers import torch
from paper_2305_16751_gb300 import domagg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("values0,values1,by_nodes", [(2, 2, False), (900, 900, False), (2, 1 << 24, False),
                                                     (1 << 24, 40, False), (1 << 24, 1 << 24, True),
                                                     (900, 1 << 24, True)])
def test_route_by_distinct_values(values0, values1, by_nodes):
    t = torch()
    g = t.Generator(device="cuda").manual_seed(10250)
    n = 300000
    D, Q = (t.randint(0, 1 << 24, (n, 3), dtype=t.int32, device="cuda", generator=g) for _ in range(2))
    for x in (D, Q):
        x[:, 0] %= values0
        x[:, 1] %= values1
    w = t.randint(-1000, 1001, (n,), dtype=t.int64, device="cuda", generator=g)
    h = domagg.handle(0)
    outs, hbm = {}, {}
    for nodes in (1, 0, 2):
        domagg.domagg_set_tuning(h, "nodes", nodes)
        try:
            outs[nodes] = domagg.forward(D, Q, w, "sum")
        finally:
            domagg.domagg_set_tuning(h, "nodes", 1)
        st = domagg.stats()
        hbm[nodes] = st["n_records"] - st["n_records_shared"]
    assert t.equal(outs[1], outs[0]) and t.equal(outs[1], outs[2])
    assert hbm[2] < hbm[0]
    assert hbm[1] == (hbm[2] if by_nodes else hbm[0])
    qi = np.arange(0, n, 1501)
    D, Q, w = (x.cpu().numpy() for x in (D, Q, w))
    assert np.array_equal(outs[1].cpu().numpy()[qi], oracle.brute(D, Q[qi], w, "sum")[0])
