"""What the m = 3 nodes hold (their items and their own handle's workspace) is
given back when another call finds the device memory used up."""
import ctypes

import numpy as np
import pytest

from gpu_helpers import torch
from paper_2305_16751_gb300 import domagg

pytestmark = pytest.mark.gpu


def _problem(g, m, n):
    t = torch()
    D = t.randint(0, 1 << 22, (n, m), dtype=t.int32, device="cuda", generator=g)
    Q = t.randint(0, 1 << 22, (n, m), dtype=t.int32, device="cuda", generator=g)
    return D, Q, t.randint(-1000, 1001, (n,), dtype=t.int64, device="cuda", generator=g)


def _forward(h, p, out):
    D, Q, w = p
    domagg.domagg_forward(h, D.shape[1], D.data_ptr(), D.shape[0], Q.data_ptr(), Q.shape[0], domagg.DTYPES["i32"],
                          w.data_ptr(), domagg.DTYPES["i64"], domagg.OPS["sum"], out.data_ptr(),
                          ctypes.c_void_p(torch().cuda.current_stream().cuda_stream))
    torch().cuda.synchronize()


def test_nodes_memory_is_given_back():
    t = torch()
    g = t.Generator(device="cuda").manual_seed(10100)
    three, two = _problem(g, 3, 1 << 21), _problem(g, 2, 12 << 20)
    out3 = t.empty(1 << 21, dtype=t.int64, device="cuda")
    out2 = t.empty(12 << 20, dtype=t.int64, device="cuda")
    # what the m = 2 call holds on a handle of its own
    h = domagg.domagg_create(0, 0)
    _forward(h, two, out2)
    want2 = out2.clone()
    need = domagg.domagg_get_stats(h)["workspace_bytes"]
    domagg.domagg_destroy(h)
    h = domagg.domagg_create(0, 0)
    try:
        _forward(h, three, out3)
        held = domagg.domagg_get_stats(h)["workspace_bytes"]
        want3 = out3.clone()
        t.cuda.synchronize()
        t.cuda.empty_cache()
        # a quarter of what the m = 2 call holds is left free: enough only
        # with what the nodes hold
        free, _ = t.cuda.mem_get_info()
        left = need // 4
        filler = t.empty(free - left, dtype=t.uint8, device="cuda")
        print("needs", need, "held", held, "left", left)
        assert held > need
        out2.zero_()
        _forward(h, two, out2)
        assert t.equal(out2, want2)
        del filler
        t.cuda.empty_cache()
        _forward(h, three, out3)
        assert t.equal(out3, want3)
    finally:
        domagg.domagg_destroy(h)
