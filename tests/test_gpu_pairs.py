"""Small problems evaluated by their definition (k_pairs) against the oracle
and against the pipeline (knob pairs = 0): tile edges, every m, operator and
non-strict mask, extreme keys, batches, plans and the flat map's statistics."""
import contextlib

import numpy as np
import pytest

import oracle
from gpu_helpers import F32_TOL, assert_matches_oracle, gpu_forward, to_dev, torch
from paper_2305_16751_gb300 import domagg, workloads

pytestmark = pytest.mark.gpu


@contextlib.contextmanager
def pipeline():
    h = domagg.handle(0)
    domagg.domagg_set_tuning(h, "pairs", 0)
    try:
        yield
    finally:
        domagg.domagg_set_tuning(h, "pairs", 1)


OPS = [("i32", "i64", "sum"), ("f32", "f32", "sum"), ("f32", "i32", "max"), ("i32", "f32", "max"),
       ("i32", "i32", "min"), ("f32", "f32", "min"), ("i32", "i64", "count")]
# query tiles of 512, stages of 128 data, several chunks of data
SIZES = ((1, 1), (127, 511), (128, 512), (129, 513), (1, 3000), (3000, 1), (5001, 4001))


@pytest.mark.parametrize("m", [1, 2, 3, 4])
@pytest.mark.parametrize("dt,wt,op", OPS)
def test_pairs_equal_oracle_and_pipeline(m, dt, wt, op):
    rng = np.random.default_rng(8100 + 10 * m + len(op) + len(wt))
    for nD, nQ in SIZES:
        for levels in (5, 900):
            D, Q, w = workloads.random_small(rng, m, nD, nQ, levels, dt, wt)
            wv = None if op == "count" else w
            got = gpu_forward(D, Q, wv, op)
            st = domagg.stats()
            assert_matches_oracle(got, D, Q, wv, op)
            with pipeline():
                ref = gpu_forward(D, Q, wv, op)
                st0 = domagg.stats()
            if not (op == "sum" and wt == "f32"):
                assert np.array_equal(got, ref)
            for key in ("n_points", "n_records", "m", "rank_bits", "distinct", "record_key_bits", "record_passes"):
                assert st[key] == st0[key], (key, nD, nQ, levels)


@pytest.mark.parametrize("m", [1, 2, 3, 4])
def test_pairs_nonstrict_and_extreme_keys(m):
    """Every mask, with the smallest and the largest int32 among the
    coordinates of both sides (a strict bound below the smallest key, a
    non-strict one at the largest)."""
    rng = np.random.default_rng(8200 + m)
    D, Q, w = workloads.random_small(rng, m, 700, 900, 6, "i32", "i64")
    for A in (D, Q):
        A[rng.random(A.shape) < 0.1] = -2**31
        A[rng.random(A.shape) < 0.1] = 2**31 - 1
    for mask in range(1 << m):
        got = domagg.forward(to_dev(D), to_dev(Q), to_dev(w), "sum", nonstrict=mask).cpu().numpy()
        want, _ = oracle.brute(D, Q, w, "sum", nonstrict=mask)
        assert np.array_equal(got, want), mask
        n = domagg.stats()["n_records"]
        with pipeline():
            domagg.forward(to_dev(D), to_dev(Q), to_dev(w), "sum", nonstrict=mask)
            assert domagg.stats()["n_records"] == n, mask


def test_pairs_backward_and_float_order():
    """The adjoint, and float sums that repeat bit for bit (fixed order of the
    chunks whatever block finishes last)."""
    rng = np.random.default_rng(8300)
    D, Q, w = workloads.random_small(rng, 3, 4000, 5000, 300, "f32", "f32")
    g = rng.standard_normal(5000).astype(np.float32)
    first = None
    for _ in range(4):
        got = domagg.backward(to_dev(D), to_dev(Q), to_dev(g)).cpu().numpy()
        first = got if first is None else first
        assert np.array_equal(got.view(np.uint32), first.view(np.uint32))
    want, S = oracle.brute_transpose(D, Q, g)
    assert np.all(np.abs(first - want) <= F32_TOL * S)


def test_pairs_cancelling_weights():
    """Weights of very different size that cancel: the float-float sum keeps
    what a plain float32 sum loses."""
    rng = np.random.default_rng(8350)
    D, Q, _ = workloads.random_small(rng, 2, 4000, 300, 4000, "i32", "f32")
    w = rng.standard_normal(4000).astype(np.float32)
    w[::2] *= np.float32(2.0**20)
    w[1::4] = -w[::4]
    D[1::4] = D[::4]
    assert_matches_oracle(gpu_forward(D, Q, w, "sum"), D, Q, w, "sum")
    want, _ = oracle.brute(D, Q, w, "sum")
    got = gpu_forward(D, Q, w, "sum").astype(np.float64)
    # one rounding of the result beside errors of order 2^-44 of the weights
    assert np.all(np.abs(got - want) <= 2.0**-24 * np.abs(want) + 4000 * 2.0**-44 * np.abs(w).max())


def test_batch_of_small_and_larger_instances():
    """Small instances by pairs beside larger ones through the pipeline, all
    m in one call; empty sides; then a NaN in a small one."""
    t = torch()
    rng = np.random.default_rng(8400)
    probs = []
    for m, nD, nQ in ((2, 60000, 50000), (3, 60000, 50000), (2, 300, 500), (3, 1000, 700), (4, 900, 1), (1, 513, 2000),
                      (2, 1, 129), (3, 600, 600), (2, 0, 40), (1, 10, 3)):
        D, Q, w = workloads.random_small(rng, m, max(nD, 1), nQ, 700, "f32", "i64")
        probs.append((D[:nD], Q, w[:nD]))
    dev = [tuple(to_dev(x) for x in p) for p in probs]
    for _ in range(2):
        outs = domagg.batch(dev, "sum")
        t.cuda.synchronize()
        for (D, Q, w), o in zip(probs, outs):
            assert_matches_oracle(o.cpu().numpy(), D, Q, w, "sum")
    dev[3][0][5, 1] = float("nan")
    for part in (dev, dev[2:4]):
        with pytest.raises(domagg.DomaggError) as e:
            domagg.batch(part, "sum")
        assert e.value.name == "NAN"
    outs = domagg.batch(dev[:3], "sum")
    assert_matches_oracle(outs[2].cpu().numpy(), *probs[2], "sum")


def test_capped_workspace_still_runs():
    """A handle whose cap leaves no room for the pairs' partials takes the
    pipeline, as long as that fits."""
    import ctypes
    t = torch()
    rng = np.random.default_rng(8500)
    D, Q, w = workloads.random_small(rng, 2, 4096, 4096, 1 << 20, "i32", "i64")
    Dd, Qd, wd = to_dev(D), to_dev(Q), to_dev(w)
    want, _ = oracle.brute(D, Q, w, "sum")
    for cap in (0, 64 << 20, 4 << 20):
        h = domagg.domagg_create(0, cap)
        try:
            out = t.zeros(4096, dtype=t.int64, device="cuda")
            domagg.domagg_forward(h, 2, Dd.data_ptr(), 4096, Qd.data_ptr(), 4096, domagg.DTYPES["i32"], wd.data_ptr(),
                                  domagg.DTYPES["i64"], domagg.OPS["sum"], out.data_ptr(),
                                  ctypes.c_void_p(t.cuda.current_stream().cuda_stream))
            assert np.array_equal(out.cpu().numpy(), want), cap
        finally:
            domagg.domagg_destroy(h)
