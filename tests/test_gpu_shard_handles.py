"""Shards of one forward on different handles: the split of the flat map
depends on the data and the knobs only, not on a handle's workspace cap."""
import ctypes

import numpy as np
import pytest

from gpu_helpers import gpu_forward, to_dev, torch
from paper_2305_16751_gb300 import domagg, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,nD,nQ", [(2, 20000, 15000), (2, 200000, 150000), (3, 20000, 15000), (3, 60000, 50000)])
@pytest.mark.parametrize("nshards", [2, 3])
def test_capped_and_uncapped_handles_split_alike(m, nD, nQ, nshards):
    t = torch()
    rng = np.random.default_rng(9990 + m)
    D, Q, w = workloads.random_small(rng, m, nD, nQ, 1 << 20, "f32", "i64")
    whole = gpu_forward(D, Q, w, "sum")
    Dd, Qd, wd = to_dev(D), to_dev(Q), to_dev(w)
    s = ctypes.c_void_p(t.cuda.current_stream().cuda_stream)
    handles = [domagg.domagg_create(0, cap) for cap in (0, 8 << 30)]
    try:
        for first in (0, 1):
            parts = []
            for shard in range(nshards):
                h = handles[(first + shard) % 2]
                out = t.zeros(nQ, dtype=t.int64, device="cuda")
                domagg._check(h, domagg.lib().domagg_forward_shard(
                    h, shard, nshards, m, Dd.data_ptr(), nD, Qd.data_ptr(), nQ, domagg.DTYPES["f32"], wd.data_ptr(),
                    domagg.DTYPES["i64"], domagg.OPS["sum"], out.data_ptr(), None, s))
                t.cuda.synchronize()
                parts.append(out)
            got = sum(parts).cpu().numpy()
            assert np.array_equal(got, whole), (first, np.count_nonzero(got != whole))
    finally:
        for h in handles:
            domagg.domagg_destroy(h)
