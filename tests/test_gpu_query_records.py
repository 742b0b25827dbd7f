"""n_query_records of calls by pairs: for m = 1 and m = 4, where the pipeline
counts every query's records, the pipeline's figure."""
import numpy as np
import pytest

from gpu_helpers import to_dev, torch
from paper_2305_16751_gb300 import domagg, workloads

pytestmark = pytest.mark.gpu


def _both(run):
    h = domagg.handle(0)
    run()
    got = domagg.stats()
    domagg.domagg_set_tuning(h, "pairs", 0)
    try:
        run()
        return got, domagg.stats()
    finally:
        domagg.domagg_set_tuning(h, "pairs", 1)


@pytest.mark.parametrize("m", [1, 4])
@pytest.mark.parametrize("nD,nQ", [(1, 1), (0, 300), (513, 700), (6000, 5001), (12000, 12000)])
def test_query_records_equal_the_pipelines(m, nD, nQ):
    rng = np.random.default_rng(10500 + m)
    D, Q, w = workloads.random_small(rng, m, max(nD, 1), nQ, 300, "i32", "i64")
    D, Q, w = to_dev(D[:nD]), to_dev(Q), to_dev(w[:nD])
    for mask in (0, 1, (1 << m) - 1):
        got, ref = _both(lambda: domagg.forward(D, Q, w, "sum", nonstrict=mask))
        assert got["n_query_records"] == ref["n_query_records"], mask


@pytest.mark.parametrize("m", [1, 4])
def test_query_records_of_a_batch(m):
    rng = np.random.default_rng(10600 + m)
    probs = [tuple(to_dev(x) for x in workloads.random_small(rng, m, 400 * i + 1, 300 * i + 2, 90, "i32", "i64"))
             for i in range(5)]
    got, ref = _both(lambda: domagg.batch(probs, "sum"))
    assert got["n_query_records"] == ref["n_query_records"]
    probs.append(tuple(to_dev(x) for x in workloads.random_small(rng, m, 20000, 15000, 900, "i32", "i64")))
    got, ref = _both(lambda: domagg.batch(probs, "sum"))
    assert got["n_query_records"] == ref["n_query_records"]
    torch().cuda.synchronize()
