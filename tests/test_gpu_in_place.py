"""Outputs that share memory with inputs (out == d_weights, grad_w ==
grad_out, an instance's output that is another's weights), at sizes that
otherwise go by pairs: every input is read before an output is written."""
import ctypes

import numpy as np
import pytest

import oracle
from gpu_helpers import F32_TOL, assert_matches_oracle, to_dev, torch
from paper_2305_16751_gb300 import domagg, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [700, 6000, 12000])
@pytest.mark.parametrize("wt,op", [("i64", "sum"), ("f32", "sum"), ("i32", "max"), ("f32", "min")])
def test_forward_into_its_weights(m, n, wt, op):
    rng = np.random.default_rng(9900 + m + n)
    D, Q, w = workloads.random_small(rng, m, n, n, 4000, "f32", wt)
    buf = to_dev(w)
    domagg.forward(to_dev(D), to_dev(Q), buf, op, out=buf)
    assert_matches_oracle(buf.cpu().numpy(), D, Q, w, op)


def test_forward_into_its_coordinates():
    rng = np.random.default_rng(9950)
    D, Q, w = workloads.random_small(rng, 1, 9000, 9000, 4000, "i32", "i32")
    for which in (0, 1):
        c = [to_dev(D), to_dev(Q)]
        out = c[which].view(-1)
        domagg.forward(c[0], c[1], to_dev(w), "max", out=out)
        assert_matches_oracle(out.cpu().numpy(), D, Q, w, "max")


def test_backward_into_its_gradient():
    rng = np.random.default_rng(9960)
    D, Q, _ = workloads.random_small(rng, 3, 8000, 8000, 3000, "f32", "f32")
    g = rng.standard_normal(8000).astype(np.float32)
    Dd, Qd, buf = to_dev(D), to_dev(Q), to_dev(g)
    domagg.domagg_backward(domagg.handle(0), 3, Dd.data_ptr(), 8000, Qd.data_ptr(), 8000, domagg.DTYPES["f32"],
                           buf.data_ptr(), buf.data_ptr(), ctypes.c_void_p(torch().cuda.current_stream().cuda_stream))
    want, S = oracle.brute_transpose(D, Q, g)
    assert np.all(np.abs(buf.cpu().numpy() - want) <= F32_TOL * S)


def _chain(rng, m, n, k):
    """k problems of n points per side; instance i's output is instance
    i + 1's weights."""
    host = [workloads.random_small(rng, m, n, n, 500, "i32", "i64") for _ in range(k)]
    dev = [[to_dev(x) for x in p] for p in host]
    arr, outs, _ = domagg._instances(dev, "sum")
    for i in range(k - 1):
        arr[i].out = arr[i + 1].d_weights
    return host, dev, arr, outs[-1]


@pytest.mark.parametrize("planned", [False, True])
def test_batch_outputs_are_weights(planned):
    rng = np.random.default_rng(9970)
    t = torch()
    host, dev, arr, last = _chain(rng, 2, 5000, 6)
    s = ctypes.c_void_p(t.cuda.current_stream().cuda_stream)
    dt = (domagg.DTYPES["i32"], domagg.DTYPES["i64"], domagg.OPS["sum"])
    plan = domagg.domagg_batch_plan(0, 6, arr, *dt, 0.5, s) if planned else None
    try:
        for (_, _, w), d in zip(host, dev):  # (planning has run the batch)
            d[2].copy_(to_dev(w))
        if planned:
            domagg.domagg_plan_run(plan, s)
            domagg.domagg_plan_status(plan, s)
        else:
            domagg.domagg_batch(domagg.handle(0), 6, arr, *dt, s)
        t.cuda.synchronize()
    finally:
        if planned:
            domagg.domagg_plan_destroy(plan)
    for i in range(6):
        got = (dev[i + 1][2] if i < 5 else last).cpu().numpy()
        assert np.array_equal(got, oracle.brute(*host[i], "sum")[0]), i
