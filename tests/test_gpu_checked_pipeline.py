"""The checked build (every computed index tested) on the pipeline's own
paths: with pairs = 0 the m = 1 scan, the groups, tiles and records of m = 2,
the pairs inside groups of m = 3 with its records and its nodes, m = 4,
overflowing groups, batches, plans, shards, the backward and the fixed
scratch; status OK and results equal to the oracle's."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import ctypes
import numpy as np, torch, oracle
from paper_2305_16751_gb300 import domagg, workloads
assert "checked" in domagg.domagg_version(), domagg.domagg_version()
rng = np.random.default_rng(52)
dev = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).cuda()
clean = lambda: domagg.domagg_sync_status(domagg.handle(0), None)

def tied(m, nD, nQ, levels, tie):
    D, Q, w = workloads.random_small(rng, m, nD, nQ, levels, "i32", "i64")
    D[:tie, 0] = 0
    Q[:tie, 0] = 0
    return D, Q, w

for m in (1, 2, 3, 4):
    for nD, nQ, levels in ((9001, 7003, 7), (9001, 7003, 1 << 20), (1, 5000, 50), (4096, 4097, 300)):
        if m == 4 and levels > 1000:
            levels = 1000
        D, Q, w = workloads.random_small(rng, m, nD, nQ, levels, "i32", "i64")
        for op, ww in (("sum", w), ("sum", w.astype(np.float32)), ("count", None), ("max", w.astype(np.int32))):
            for mask in (0, (1 << m) - 1):
                got = domagg.forward(dev(D), dev(Q), dev(ww), op, nonstrict=mask).cpu().numpy()
                want, _ = oracle.brute(D, Q, ww, op, nonstrict=mask)
                assert np.array_equal(got.astype(np.int64), want.astype(np.int64)), (m, nD, levels, op, mask)
        clean()
    if m in (2, 3):
        D, Q, w = tied(m, 40000, 31000, 1 << 20, 8000)
        got = domagg.forward(dev(D), dev(Q), dev(w), "sum").cpu().numpy()
        assert np.array_equal(got, oracle.brute(D, Q, w, "sum")[0]), m
        D, Q, w = tied(m, 20000, 16000, 1 << 20, 8000)  # no group width qualifies
        got = domagg.forward(dev(D), dev(Q), dev(w), "sum").cpu().numpy()
        assert np.array_equal(got, oracle.brute(D, Q, w, "sum")[0]), m
        parts = [domagg.forward_shard(dev(D), dev(Q), dev(w), "sum", s, 3)[0] for s in range(3)]
        assert np.array_equal(domagg.combine(parts, None, "sum", torch.int64).cpu().numpy(), got), m
    D, Q, _ = workloads.random_small(rng, m, 6000, 5000, 900, "i32", "i64")
    g = rng.integers(-9, 10, size=5000).astype(np.float32)
    gw = domagg.backward(dev(D), dev(Q), dev(g)).cpu().numpy()
    assert np.array_equal(gw.astype(np.float64), oracle.brute_transpose(D, Q, g)[0]), m
    clean()

probs = [workloads.random_small(rng, 1 + i % 4, 300 + 700 * i, 2500, 60, "i32", "i64") for i in range(9)]
probs.append(tied(3, 40000, 31000, 1 << 20, 8000))
want = [oracle.brute(D, Q, w, "sum")[0] for D, Q, w in probs]
pd = [tuple(dev(x) for x in p) for p in probs]
for _ in range(2):
    for o, v in zip(domagg.batch(pd, "sum"), want):
        assert np.array_equal(o.cpu().numpy(), v)
plan = domagg.BatchPlan(pd, "sum", headroom=0.2)
for _ in range(2):
    plan.run()
    plan.status()
    for o, v in zip(plan.outs, want):
        assert np.array_equal(o.cpu().numpy(), v)
plan.close()

D, Q, w = workloads.random_small(rng, 3, 9000, 8000, 3000, "i32", "i64")
Dd, Qd, wd = dev(D), dev(Q), dev(w)
out = torch.empty(8000, dtype=torch.int64, device="cuda")
st = domagg.lib().domagg_forward_noalloc(3, Dd.data_ptr(), 9000, Qd.data_ptr(), 8000, 0, wd.data_ptr(), 1, 0,
                                         out.data_ptr(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
torch.cuda.synchronize()
assert st == 0 and np.array_equal(out.cpu().numpy(), oracle.brute(D, Q, w, "sum")[0])
clean()
print("CHECKED OK")
"""


@pytest.mark.parametrize("nodes", [0, 2])
def test_checked_build_runs_the_pipeline_clean(nodes):
    env = dict(os.environ, DOMAGG_CHECKED="1", PYTHONPATH=ROOT, DOMAGG_TUNE=f"pairs=0,nodes={nodes}")
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, env=env, capture_output=True, text=True,
                       timeout=900)
    assert r.returncode == 0 and "CHECKED OK" in r.stdout, r.stdout[-2000:] + r.stderr[-4000:]
