"""m = 3 groups of ranks by level walks (k_walk3; knob walk3 = 2 takes them
always): the groups' and the nodes' tests once more with them, the checked
build, and the rule that takes them where the coordinates have few distinct
values and the groups fill the chip."""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
import test_gpu_checked_pipeline
import test_gpu_groups3
import test_gpu_nodes
from gpu_helpers import F32_TOL, assert_matches_oracle, gpu_forward, to_dev, torch
from paper_2305_16751_gb300 import domagg, workloads

pytestmark = pytest.mark.gpu

for _mod in (test_gpu_groups3, test_gpu_nodes):
    for _name, _fn in list(vars(_mod).items()):
        if _name.startswith("test_") and callable(_fn) and _name != "test_batch_in_parts_equals_single_calls":
            globals()[_name] = _fn


@pytest.fixture(autouse=True)
def walks(monkeypatch):
    h = domagg.handle(0)
    monkeypatch.setenv("DOMAGG_TUNE", "walk3=2")
    domagg.domagg_set_tuning(h, "walk3", 2)
    yield
    domagg.domagg_set_tuning(h, "walk3", 1)


CASES = [("i32", "i64", "sum"), ("f32", "f32", "sum"), ("f32", "i32", "max"), ("i32", "f32", "min"),
         ("f32", "i64", "count")]


@pytest.mark.parametrize("dt,wt,op", CASES)
def test_walks_equal_oracle_and_pairs(dt, wt, op):
    """Tile and group edges (5120 and 10240 points a group), one value, few
    values, many; small blocks taken by pairs inside the walk."""
    rng = np.random.default_rng(11200 + len(op) + len(wt))
    h = domagg.handle(0)
    domagg.domagg_set_tuning(h, "pairs", 0)
    try:
        for nD, nQ, levels in ((1, 1, 1), (2560, 2560, 3), (2560, 2561, 40), (5120, 5120, 40), (5120, 5121, 40),
                               (15000, 9000, 200), (9000, 15000, 2), (7000, 6000, 1 << 20), (3, 4000, 9)):
            D, Q, w = workloads.random_small(rng, 3, nD, nQ, levels, dt, wt)
            wv = None if op == "count" else w
            got = gpu_forward(D, Q, wv, op)
            assert_matches_oracle(got, D, Q, wv, op)
            domagg.domagg_set_tuning(h, "walk3", 0)
            ref = gpu_forward(D, Q, wv, op)
            domagg.domagg_set_tuning(h, "walk3", 2)
            if not (op == "sum" and wt == "f32"):
                assert np.array_equal(got, ref), (nD, nQ, levels)
    finally:
        domagg.domagg_set_tuning(h, "pairs", 1)


def test_walks_float_sums_repeat_and_backward():
    rng = np.random.default_rng(11300)
    D, Q, w = workloads.random_small(rng, 3, 60000, 50000, 60, "f32", "f32")
    Dd, Qd, wd = to_dev(D), to_dev(Q), to_dev(w)
    a, b = (domagg.forward(Dd, Qd, wd, "sum").cpu().numpy() for _ in range(2))
    assert np.array_equal(a.view(np.uint32), b.view(np.uint32))
    qi = np.arange(0, 50000, 23)
    want, S = oracle.brute(D, Q[qi], w, "sum")
    assert np.all(np.abs(a[qi].astype(np.float64) - want) <= F32_TOL * S)
    g = rng.standard_normal(50000).astype(np.float32)
    got = domagg.backward(Dd, Qd, to_dev(g)).cpu().numpy()
    di = np.arange(0, 60000, 23)
    want, S = oracle.brute_transpose(D[di], Q, g)
    assert np.all(np.abs(got[di] - want) <= F32_TOL * S)


@pytest.mark.parametrize("k,n,values,by_walks", [(100, 8000, 40, True), (24, 40000, 200, True), (60, 8000, 1 << 22, False),
                                                (1, 20000, 40, False)])
def test_rule(monkeypatch, k, n, values, by_walks):
    """The statistics of the route the rule takes are the walks' or the pairs'
    (their groups differ), and plans choose like calls."""
    t = torch()
    g = t.Generator(device="cuda").manual_seed(11400 + k)
    probs = []
    for _ in range(k):
        D, Q = (t.randint(0, values, (n, 3), dtype=t.int32, device="cuda", generator=g) for _ in range(2))
        probs.append((D, Q, t.randint(-1000, 1001, (n,), dtype=t.int64, device="cuda", generator=g)))
    h = domagg.handle(0)
    outs, shared = {}, {}
    domagg.domagg_set_tuning(h, "nodes", 0)
    try:
        for mode in (0, 2, 1):
            domagg.domagg_set_tuning(h, "walk3", mode)
            outs[mode] = domagg.batch(probs, "sum")
            shared[mode] = domagg.stats()["n_records_shared"]
    finally:
        domagg.domagg_set_tuning(h, "nodes", 1)
    assert shared[0] != shared[2]
    assert shared[1] == shared[2 if by_walks else 0]
    monkeypatch.setenv("DOMAGG_TUNE", "walk3=1")
    plan = domagg.BatchPlan(probs, "sum", headroom=0.1)
    try:
        plan.run()
        plan.status()
        for o, a, b, c in zip(plan.outs, outs[0], outs[1], outs[2]):
            assert t.equal(a, b) and t.equal(a, c) and t.equal(a, o)
    finally:
        plan.close()
    D, Q, w = (x.cpu().numpy() for x in probs[0])
    qi = np.arange(0, n, 97)
    assert np.array_equal(outs[1][0].cpu().numpy()[qi], oracle.brute(D, Q[qi], w, "sum")[0])


@pytest.mark.parametrize("nodes", [0, 2])
def test_checked_build_walks_clean(nodes):
    env = dict(os.environ, DOMAGG_CHECKED="1", PYTHONPATH=test_gpu_checked_pipeline.ROOT,
               DOMAGG_TUNE=f"pairs=0,walk3=2,nodes={nodes}")
    r = subprocess.run([sys.executable, "-c", test_gpu_checked_pipeline.SCRIPT], cwd=test_gpu_checked_pipeline.ROOT,
                       env=env, capture_output=True, text=True, timeout=900)
    assert r.returncode == 0 and "CHECKED OK" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
