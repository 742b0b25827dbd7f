"""The pipeline at sizes that go by pairs by default: the parity tests of the
forward, the backward, batches, variants and plans once more with the knob
pairs = 0, and for m = 3 with the levels above the groups by records
(nodes = 0) and by nodes (nodes = 2).  The knobs reach the shared handle, and
through DOMAGG_TUNE the handles that plans and other tests create."""
import numpy as np
import pytest

import oracle
import test_gpu_backward_batch
import test_gpu_forward
import test_gpu_plan
import test_gpu_variants
from gpu_helpers import assert_matches_oracle, to_dev, torch
from paper_2305_16751_gb300 import domagg, workloads

pytestmark = pytest.mark.gpu

LARGE = ("test_batch_full_recipe_sampled", "test_basic_variant_at_scale_m2",
         "test_plan_autotune_with_ranges_of_top_levels")
for _mod in (test_gpu_forward, test_gpu_backward_batch, test_gpu_variants, test_gpu_plan):
    for _name, _fn in list(vars(_mod).items()):
        if _name.startswith("test_") and callable(_fn) and _name not in LARGE:
            globals()[_name] = _fn


@pytest.fixture(autouse=True, params=[0, 2], ids=["records", "nodes"])
def pipeline(request, monkeypatch):
    h = domagg.handle(0)
    monkeypatch.setenv("DOMAGG_TUNE", f"pairs=0,nodes={request.param}")
    domagg.domagg_set_tuning(h, "pairs", 0)
    domagg.domagg_set_tuning(h, "nodes", request.param)
    yield
    domagg.domagg_set_tuning(h, "pairs", 1)
    domagg.domagg_set_tuning(h, "nodes", 1)


def _extremes(rng, A):
    A[rng.random(A.shape) < 0.1] = -2**31
    A[rng.random(A.shape) < 0.1] = 2**31 - 1


@pytest.mark.parametrize("mask", range(16))
def test_m4_every_mask_and_extreme_keys(mask):
    rng = np.random.default_rng(10700 + mask)
    D, Q, w = workloads.random_small(rng, 4, 2600, 2300, 40, "i32", "i64")
    _extremes(rng, D)
    _extremes(rng, Q)
    got = domagg.forward(to_dev(D), to_dev(Q), to_dev(w), "sum", nonstrict=mask).cpu().numpy()
    assert np.array_equal(got, oracle.brute(D, Q, w, "sum", nonstrict=mask)[0])


@pytest.mark.parametrize("mask", range(8))
def test_m3_every_mask_and_extreme_keys(mask):
    rng = np.random.default_rng(10800 + mask)
    D, Q, w = workloads.random_small(rng, 3, 16000, 9000, 3000, "i32", "i64")
    _extremes(rng, D)
    _extremes(rng, Q)
    got = domagg.forward(to_dev(D), to_dev(Q), to_dev(w), "sum", nonstrict=mask).cpu().numpy()
    assert np.array_equal(got, oracle.brute(D, Q, w, "sum", nonstrict=mask)[0])


@pytest.mark.parametrize("op,wt", [("sum", "f32"), ("sum", "i64"), ("max", "i32"), ("min", "f32"), ("count", "i64")])
def test_planned_m4_replayed_with_new_data(op, wt):
    t = torch()
    rng = np.random.default_rng(10900)
    host, levels = [], []
    for m, nD, nQ, lv in ((4, 3000, 2500, 50), (3, 9000, 7000, 900), (4, 700, 900, 300), (2, 4000, 4100, 70),
                          (1, 5000, 4000, 1000)):
        host.append(workloads.random_small(rng, m, nD, nQ, lv, "i32", wt))
        levels.append(lv)
    dev = [tuple(to_dev(x) for x in p) for p in host]
    plan = domagg.BatchPlan(dev, op, headroom=0.5)
    try:
        g = t.cuda.CUDAGraph()
        side = t.cuda.Stream()
        side.wait_stream(t.cuda.current_stream())
        with t.cuda.stream(side):
            with t.cuda.graph(g, stream=side):
                plan.run()
        t.cuda.synchronize()
        for _ in range(2):
            host = test_gpu_plan._refill(rng, dev, host, levels, wt)
            g.replay()
            plan.status()
            for (D, Q, w), o in zip(host, plan.outs):
                assert_matches_oracle(o.cpu().numpy(), D, Q, None if op == "count" else w, op)
    finally:
        plan.close()
