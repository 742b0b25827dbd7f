"""m = 1 by the scan over the permutation (k_line): tile edges (4096 points),
ties, both comparisons, every operator, batches and plans, against the
oracle; float sums repeat bit for bit."""
import os

import numpy as np
import pytest

import oracle
from gpu_helpers import F32_TOL, assert_matches_oracle, gpu_forward, to_dev, torch
from paper_2305_16751_gb300 import domagg, workloads

pytestmark = pytest.mark.gpu

OPS = [("i32", "i64", "sum"), ("f32", "f32", "sum"), ("f32", "i32", "max"), ("i32", "f32", "min"),
       ("f32", "i64", "count")]


@pytest.fixture(autouse=True)
def pipeline():
    h = domagg.handle(0)
    domagg.domagg_set_tuning(h, "pairs", 0)
    yield
    domagg.domagg_set_tuning(h, "pairs", 1)


@pytest.mark.parametrize("dt,wt,op", OPS)
def test_line_equals_oracle(dt, wt, op):
    rng = np.random.default_rng(9500 + len(op) + len(wt))
    for nD, nQ in ((1, 1), (2048, 2047), (2048, 2048), (2049, 2048), (0, 5000), (30001, 27003), (5000, 1)):
        for levels in (3, 100000):
            D, Q, w = workloads.random_small(rng, 1, max(nD, 1), nQ, levels, dt, wt)
            D, w = D[:nD], w[:nD]
            wv = None if op == "count" else w
            assert_matches_oracle(gpu_forward(D, Q, wv, op), D, Q, wv, op)
            assert domagg.stats()["n_records"] == nD + nQ
            want, S = oracle.brute(D, Q, wv, op, nonstrict=1)
            got = domagg.forward(to_dev(D), to_dev(Q), to_dev(wv), op, nonstrict=1).cpu().numpy()
            assert_matches_oracle(got, D, Q, wv, op, want=want, S=S)


def test_line_float_sums_repeat_and_backward():
    rng = np.random.default_rng(9600)
    D, Q, w = workloads.random_small(rng, 1, 300000, 250000, 5000, "f32", "f32")
    Dd, Qd, wd = to_dev(D), to_dev(Q), to_dev(w)
    a, b = (domagg.forward(Dd, Qd, wd, "sum").cpu().numpy() for _ in range(2))
    assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
    qi = rng.integers(0, 250000, size=2000)
    want, S = oracle.brute(D, Q[qi], w, "sum")
    assert np.all(np.abs(a[qi].astype(np.float64) - want) <= F32_TOL * S)
    g = rng.standard_normal(9000).astype(np.float32)
    got = domagg.backward(to_dev(D[:7000]), to_dev(Q[:9000]), to_dev(g)).cpu().numpy()
    want, S = oracle.brute_transpose(D[:7000], Q[:9000], g)
    assert np.all(np.abs(got - want) <= F32_TOL * S)


def test_line_in_batches_and_plans():
    t = torch()
    rng = np.random.default_rng(9700)
    probs = [workloads.random_small(rng, 1, int(n), int(n) + 7, 900, "i32", "i64") for n in (9000, 1, 4096, 12000)]
    dev = [tuple(to_dev(x) for x in p) for p in probs]
    outs = domagg.batch(dev, "sum")
    os.environ["DOMAGG_TUNE"] = "pairs=0"
    try:
        plan = domagg.BatchPlan(dev, "sum")
    finally:
        del os.environ["DOMAGG_TUNE"]
    try:
        plan.run()
        plan.status()
        for (D, Q, w), o, po in zip(probs, outs, plan.outs):
            want, _ = oracle.brute(D, Q, w, "sum")
            assert np.array_equal(o.cpu().numpy(), want) and t.equal(o, po)
    finally:
        plan.close()
