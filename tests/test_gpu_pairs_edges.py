"""Small problems by pairs at the edges of k_pairs' stages (512 data), of the
statistics' forms (8192 points: 256 or 1024 threads per block; in a batch 2, 8
or 24 items per thread by its largest instance) and of the route itself
(24576 points), against the oracle and the pipeline's statistics."""
import numpy as np
import pytest

from gpu_helpers import assert_matches_oracle, to_dev, torch
from paper_2305_16751_gb300 import domagg, workloads

pytestmark = pytest.mark.gpu

KEYS = ("n_points", "n_records", "m")


def _both(run):
    h = domagg.handle(0)
    outs = run()
    st = domagg.stats()
    domagg.domagg_set_tuning(h, "pairs", 0)
    try:
        refs = run()
        return outs, st, refs, domagg.stats()
    finally:
        domagg.domagg_set_tuning(h, "pairs", 1)


@pytest.mark.parametrize("m", [1, 2, 3, 4])
@pytest.mark.parametrize("nD,nQ", [(511, 600), (512, 600), (513, 513), (1024, 511), (1025, 512), (4096, 4096),
                                   (4097, 4096), (12288, 12288), (12288, 12289)])
def test_stage_and_route_edges(m, nD, nQ):
    rng = np.random.default_rng(11000 + m + nD)
    D, Q, w = workloads.random_small(rng, m, nD, nQ, 700, "f32", "i64")
    Dd, Qd, wd = to_dev(D), to_dev(Q), to_dev(w)
    out, st, ref, st0 = _both(lambda: domagg.forward(Dd, Qd, wd, "sum"))
    assert torch().equal(out, ref)
    for key in KEYS + ("rank_bits", "distinct", "record_key_bits"):
        assert st[key] == st0[key], key
    qi = np.arange(0, nQ, max(1, nQ // 700))
    assert_matches_oracle(out.cpu().numpy(), D, Q, w, "sum", qidx=qi)


@pytest.mark.parametrize("m", [2, 3, 4])
@pytest.mark.parametrize("largest", [2048, 2049, 8192, 8193, 24576])
@pytest.mark.parametrize("mask_levels", [7, 5000])
def test_statistics_of_a_batch(m, largest, mask_levels):
    rng = np.random.default_rng(11100 + m + largest)
    probs = []
    for n in (largest, 2, 1000, largest // 2 + 1, 511):
        nQ = max(1, n // 3)
        probs.append(workloads.random_small(rng, m, n - nQ, nQ, mask_levels, "i32", "i64"))
    dev = [tuple(to_dev(x) for x in p) for p in probs]
    outs, st, refs, st0 = _both(lambda: domagg.batch(dev, "sum"))
    for key in KEYS:
        assert st[key] == st0[key], key
    for (D, Q, w), o, r in zip(probs, outs, refs):
        assert torch().equal(o, r)
        assert_matches_oracle(o.cpu().numpy(), D, Q, w, "sum", qidx=np.arange(0, Q.shape[0], 1 + Q.shape[0] // 300))
