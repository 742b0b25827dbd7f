"""Workspace caps: what a small call held must not keep a larger call from the
room it has on a fresh handle with the same cap."""
import contextlib
import ctypes

import numpy as np
import pytest

from gpu_helpers import to_dev, torch
from paper_2305_16751_gb300 import domagg, workloads

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def capped(cap, pairs=1):
    h = domagg.domagg_create(0, cap)
    domagg.domagg_set_tuning(h, "pairs", pairs)
    try:
        yield h
    finally:
        domagg.domagg_destroy(h)


def _stream():
    return ctypes.c_void_p(torch().cuda.current_stream().cuda_stream)


def _forward(h, p):
    D, Q, w = p
    out = torch().zeros(Q.shape[0], dtype=torch().int64, device="cuda")
    domagg.domagg_forward(h, D.shape[1], D.data_ptr(), D.shape[0], Q.data_ptr(), Q.shape[0], domagg.DTYPES["i32"],
                          w.data_ptr(), domagg.DTYPES["i64"], domagg.OPS["sum"], out.data_ptr(), _stream())
    torch().cuda.synchronize()
    return out


def _batch(h, probs):
    arr, outs, _ = domagg._instances(probs, "sum")
    domagg.domagg_batch(h, len(probs), arr, domagg.DTYPES["i32"], domagg.DTYPES["i64"], domagg.OPS["sum"], _stream())
    torch().cuda.synchronize()
    return outs


def _smallest_cap(run, pairs):
    """The smallest cap (to 64 KiB) with which run works on a fresh handle."""
    lo, hi = 0, 1 << 30
    while hi - lo > 1 << 16:
        mid = (lo + hi) // 2
        with capped(mid, pairs) as h:
            try:
                run(h)
                hi = mid
            except domagg.DomaggError as e:
                assert e.name == "OOM"
                lo = mid
    return hi


def _dev(rng, m, nD, nQ, levels=1 << 20):
    return tuple(to_dev(x) for x in workloads.random_small(rng, m, nD, nQ, levels, "i32", "i64"))


@pytest.mark.parametrize("m", [2, 3])
def test_small_call_then_one_that_just_fits(m):
    rng = np.random.default_rng(10010 + m)
    small, large = _dev(rng, m, 12000, 12000), _dev(rng, m, 30000, 25000)
    cap = _smallest_cap(lambda h: _forward(h, large), 1)
    with capped(cap) as h:
        want_small, want = _forward(h, small), _forward(h, large)
        for _ in range(2):  # (and back)
            assert torch().equal(_forward(h, small), want_small)
            assert torch().equal(_forward(h, large), want)
    assert torch().equal(domagg.forward(*large, "sum"), want)
    assert torch().equal(domagg.forward(*small, "sum"), want_small)


def test_mixed_batch_that_just_fits_by_the_pipeline():
    rng = np.random.default_rng(10020)
    # the pairs' partials of the m = 3 instances: 1.6 MB
    probs = [_dev(rng, 2, 120000, 100000)] + [_dev(rng, 3, 1700, 1700) for _ in range(30)]
    cap = _smallest_cap(lambda h: _batch(h, probs), 0)
    with capped(cap) as h:
        for _ in range(2):
            outs = _batch(h, probs)
    for p, o in zip(probs, outs):
        assert torch().equal(domagg.forward(*p, "sum"), o)
