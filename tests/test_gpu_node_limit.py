"""m = 3 with more first-rank nodes than the nodes' path takes (a third of the
points on one value of the first coordinate, so that no level goes in groups,
and the rest spread): decided on the device, without running the point phase
again, for each instance by itself; results as by the records in HBM."""
import numpy as np
import pytest

import oracle
from gpu_helpers import torch
from paper_2305_16751_gb300 import domagg

pytestmark = pytest.mark.gpu


def _problem(g, n, tied):
    t = torch()
    D = t.randint(0, 1 << 24, (n, 3), dtype=t.int32, device="cuda", generator=g)
    Q = t.randint(0, 1 << 24, (n, 3), dtype=t.int32, device="cuda", generator=g)
    D[:tied, 0] = 0
    Q[:tied, 0] = 0
    return D, Q, t.randint(-1000, 1001, (n,), dtype=t.int64, device="cuda", generator=g)


def _encodes(run):
    h = domagg.handle(0)
    domagg.domagg_timing_read(h)
    domagg.domagg_timing_enable(h, True)
    try:
        outs = run()
        return outs, domagg.domagg_timing_read(h)["encode"]["launches"]
    finally:
        domagg.domagg_timing_enable(h, False)


def _by_records(run):
    h = domagg.handle(0)
    domagg.domagg_set_tuning(h, "nodes", 0)
    try:
        return run()
    finally:
        domagg.domagg_set_tuning(h, "nodes", 1)


def test_one_point_phase():
    t = torch()
    g = t.Generator(device="cuda").manual_seed(10200)
    p = _problem(g, 300000, 100000)
    out, encodes = _encodes(lambda: domagg.forward(*p, "sum"))
    assert encodes == 1
    assert t.equal(out, _by_records(lambda: domagg.forward(*p, "sum")))
    D, Q, w = (x.cpu().numpy() for x in p)
    qi = np.arange(0, 300000, 1501)
    assert np.array_equal(out.cpu().numpy()[qi], oracle.brute(D, Q[qi], w, "sum")[0])


def test_instances_decide_by_themselves():
    """Beside an instance with too many nodes, others keep theirs."""
    t = torch()
    g = t.Generator(device="cuda").manual_seed(10300)
    probs = [_problem(g, 150000, 50000), _problem(g, 200000, 0), _problem(g, 40000, 0), _problem(g, 100000, 30000)]
    outs, encodes = _encodes(lambda: domagg.batch(probs, "sum"))
    assert encodes == 1
    shared = domagg.stats()["n_records_shared"]
    want = _by_records(lambda: domagg.batch(probs, "sum"))
    assert shared > domagg.stats()["n_records_shared"]
    for o, v in zip(outs, want):
        assert t.equal(o, v)
