"""Calls on one handle that follow each other without a synchronisation: a
call returns with the upload of its record tables still queued behind its
kernels, and the next call's tables, of another number of instances, go to
the same pinned area.  Every first call here has records in HBM (more points
on one value of the first coordinate than a group holds)."""
import numpy as np
import pytest

from gpu_helpers import torch
from paper_2305_16751_gb300 import domagg

pytestmark = pytest.mark.gpu


def _problem(g, m, nD, nQ, levels=1 << 20, tie=0):
    t = torch()
    D = t.randint(0, levels, (nD, m), dtype=t.int32, device="cuda", generator=g)
    Q = t.randint(0, levels, (nQ, m), dtype=t.int32, device="cuda", generator=g)
    if tie:
        D[:tie, 0] = 5
        Q[:tie, 0] = 5
    w = t.randint(-1000, 1001, (nD,), dtype=t.int64, device="cuda", generator=g)
    return D, Q, w


def _singles(probs):
    outs = []
    for p in probs:
        outs.append(domagg.forward(*p, "sum"))
        torch().cuda.synchronize()
    return outs


def _equal(outs, want, what):
    torch().cuda.synchronize()
    for i, (o, v) in enumerate(zip(outs, want)):
        assert torch().equal(o, v), (what, i)


@pytest.mark.parametrize("m", [2, 3])
@pytest.mark.parametrize("k1,k2", [(3, 4), (3, 6), (8, 10), (8, 24)])
def test_batch_after_batch(m, k1, k2):
    g = torch().Generator(device="cuda").manual_seed(9600 + 100 * m + k1 + k2)
    first = [_problem(g, m, 130000, 110000, tie=9000) for _ in range(k1)]
    second = [_problem(g, m, 20000 + 100 * i, 15000) for i in range(k2)]
    want1, want2 = _singles(first), _singles(second)
    for _ in range(3):
        outs1 = domagg.batch(first, "sum")
        assert domagg.stats()["n_records_shared"] < domagg.stats()["n_records"]
        outs2 = domagg.batch(second, "sum")
        _equal(outs1, want1, "first")
        _equal(outs2, want2, "second")


def test_halves_of_a_mixed_batch():
    """The m = 2 instances' call, then the m = 3 instances', in one batch."""
    g = torch().Generator(device="cuda").manual_seed(9700)
    probs = [_problem(g, 2, 300000, 250000, tie=9000) for _ in range(4)]
    probs += [_problem(g, 3, 20000, 15000 + 100 * i) for i in range(8)]
    want = _singles(probs)
    for _ in range(3):
        _equal(domagg.batch(probs, "sum"), want, "mixed")


def test_parts_of_a_large_batch():
    """m = 3, more than 2^25 points: a first part of three instances with
    records in HBM, a second of six."""
    g = torch().Generator(device="cuda").manual_seed(9800)
    probs = [_problem(g, 3, 6_000_000, 5_150_000, levels=1 << 22, tie=9000) for _ in range(3)]
    probs += [_problem(g, 3, 70000, 60000) for _ in range(6)]
    assert sum(p[0].shape[0] + p[1].shape[0] for p in probs[:4]) > 1 << 25
    want = _singles(probs)
    for _ in range(2):
        _equal(domagg.batch(probs, "sum"), want, "parts")
