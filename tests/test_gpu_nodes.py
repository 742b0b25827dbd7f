"""m = 3: the first rank's levels above the groups as m = 2 problems, one per
node (knob nodes = 2 at small sizes), against the oracle and against the
records in HBM (nodes = 0); with groups, without them, and with groups too
large for pairs; item tiles of 4096 and their edges."""
import contextlib

import numpy as np
import pytest

import oracle
from gpu_helpers import F32_TOL, assert_matches_oracle, gpu_forward, to_dev, torch
from paper_2305_16751_gb300 import domagg, workloads

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def knobs(**kw):
    h = domagg.handle(0)
    defaults = {"pairs": 1, "nodes": 1}
    for name, v in kw.items():
        domagg.domagg_set_tuning(h, name, v)
    try:
        yield
    finally:
        for name in kw:
            domagg.domagg_set_tuning(h, name, defaults[name])


CASES = [("i32", "i64", "sum"), ("f32", "f32", "sum"), ("f32", "i32", "max"), ("i32", "f32", "min"),
         ("f32", "i64", "count")]
# 1000 points a group on average: up to five levels above the groups
SIZES = ((30000, 20000, 1 << 20), (9001, 7003, 5000), (15000, 14000, 700), (1, 5000, 50), (5000, 1, 7),
         (3000, 3000, 2), (2048, 2048, 1 << 20), (2100, 4001, 90))


@pytest.mark.parametrize("dt,wt,op", CASES)
def test_nodes_equal_records_in_hbm(dt, wt, op):
    rng = np.random.default_rng(9100 + len(op) + len(wt))
    for nD, nQ, levels in SIZES:
        D, Q, w = workloads.random_small(rng, 3, nD, nQ, levels, dt, wt)
        wv = None if op == "count" else w
        with knobs(pairs=0, nodes=2):
            got = gpu_forward(D, Q, wv, op)
            st = domagg.stats()
        with knobs(pairs=0, nodes=0):
            ref = gpu_forward(D, Q, wv, op)
            st0 = domagg.stats()
        assert_matches_oracle(got, D, Q, wv, op)
        if not (op == "sum" and wt == "f32"):
            assert np.array_equal(got, ref), (nD, nQ, levels)
        for key in ("n_points", "n_records", "rank_bits", "distinct", "record_key_bits"):
            assert st[key] == st0[key], (key, nD, nQ, levels)
        assert st["n_records_shared"] >= st0["n_records_shared"]


@pytest.mark.parametrize("mask", range(1, 8))
def test_nodes_nonstrict(mask):
    rng = np.random.default_rng(9200 + mask)
    D, Q, w = workloads.random_small(rng, 3, 9000, 8000, 900, "f32", "i64")
    with knobs(pairs=0, nodes=2):
        got = domagg.forward(to_dev(D), to_dev(Q), to_dev(w), "sum", nonstrict=mask).cpu().numpy()
    want, _ = oracle.brute(D, Q, w, "sum", nonstrict=mask)
    assert np.array_equal(got, want)


def test_nodes_backward_batch_and_overflow():
    t = torch()
    rng = np.random.default_rng(9300)
    with knobs(pairs=0, nodes=2):
        D, Q, _ = workloads.random_small(rng, 3, 7000, 9000, 4000, "i32", "i64")
        g = rng.standard_normal(9000).astype(np.float32)
        got = domagg.backward(to_dev(D), to_dev(Q), to_dev(g)).cpu().numpy()
        want, S = oracle.brute_transpose(D, Q, g)
        assert np.all(np.abs(got - want) <= F32_TOL * S)
        probs = []
        for nD, nQ, levels in ((9000, 7000, 1 << 16), (1, 1, 2), (0, 300, 10), (777, 555, 3), (15000, 14000, 1 << 20),
                               (6000, 5000, 5), (4096, 4096, 300)):
            D, Q, w = workloads.random_small(rng, 3, max(nD, 1), nQ, levels, "i32", "i64")
            probs.append((D[:nD], Q, w[:nD]))
        outs = domagg.batch([tuple(to_dev(x) for x in p) for p in probs], "sum")
        t.cuda.synchronize()
        for (D, Q, w), o in zip(probs, outs):
            want, _ = oracle.brute(D, Q, w, "sum")
            assert np.array_equal(o.cpu().numpy(), want), (D.shape, Q.shape)
        # 11000 points on one first coordinate: that group's levels stay records
        D, Q, w = workloads.random_small(rng, 3, 40000, 31000, 1 << 20, "i32", "i64")
        D[:6000, 0] = 0
        Q[:5000, 0] = 0
        got = gpu_forward(D, Q, w, "sum")
        st = domagg.stats()
        want, _ = oracle.brute(D, Q, w, "sum")
        assert np.array_equal(got, want)
        assert 0 < st["n_records_shared"] < st["n_records"]


def test_nodes_float_sums_repeat_exactly():
    """270000 points, five levels above the groups: float32 sums repeat bit for
    bit and lie within the tolerance; int64 sums equal the records path's."""
    rng = np.random.default_rng(9400)
    D, Q, w = workloads.random_small(rng, 3, 140000, 130000, 1 << 22, "f32", "f32")
    Dd, Qd, wd = to_dev(D), to_dev(Q), to_dev(w)
    with knobs(nodes=2):
        first = domagg.forward(Dd, Qd, wd, "sum").cpu().numpy()
        again = domagg.forward(Dd, Qd, wd, "sum").cpu().numpy()
    assert np.array_equal(first.view(np.uint32), again.view(np.uint32))
    qi = rng.integers(0, 130000, size=3000)
    want, S = oracle.brute(D, Q[qi], w, "sum")
    assert np.all(np.abs(first[qi].astype(np.float64) - want) <= F32_TOL * S)
    wi = to_dev(rng.integers(-1000, 1001, size=140000))
    with knobs(nodes=2):
        got = domagg.forward(Dd, Qd, wi, "sum").cpu().numpy()
    with knobs(nodes=0):
        ref = domagg.forward(Dd, Qd, wi, "sum").cpu().numpy()
    assert np.array_equal(got, ref)


def test_batch_in_parts_equals_single_calls():
    """More points of m = 3 than one call of the nodes takes (2^25): every
    instance of the batch as its own call, bit for bit, and the statistics of
    the whole."""
    rng = np.random.default_rng(9500)
    probs = []
    for nD, nQ in ((7 << 20, 6 << 20), (4 << 20, 9 << 20), (300000, 1), (5 << 20, 5 << 20), (200000, 250000)):
        D, Q, w = workloads.random_small(rng, 3, nD, nQ, 1 << 22, "i32", "i64")
        probs.append((to_dev(D), to_dev(Q), to_dev(w)))
    points = sum(p[0].shape[0] + p[1].shape[0] for p in probs)
    assert points > 1 << 25
    outs = domagg.batch(probs, "sum")
    st = domagg.stats()
    assert st["n_points"] == points
    records = 0
    for p, o in zip(probs, outs):
        single = domagg.forward(*p, "sum")
        assert torch().equal(o, single), tuple(p[0].shape)
        records += domagg.stats()["n_records"]
    assert st["n_records"] == records
