"""Distributed shared memory: a block may store into another block of its
cluster only once every block of the cluster is known to have started, so in
every kernel a cluster barrier has to be complete before the first remote
store.  Checked on the sources (a violation is a race with a block's launch,
which no run shows reliably and which must not be run to see)."""
import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2305_16751_gb300", "csrc")


def _kernels(text):
    """(name, body) of every __global__ function of a source."""
    text = re.sub(r"//[^\n]*", "", re.sub(r"/\*.*?\*/", "", text, flags=re.S))
    for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", text):
        start = text.index("{", m.end())
        depth, i = 0, start
        while True:
            depth += {"{": 1, "}": -1}.get(text[i], 0)
            i += 1
            if depth == 0:
                break
        yield m.group(1), text[start:i]


def test_cluster_barrier_before_the_first_remote_store():
    seen = 0
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            for kernel, body in _kernels(f.read()):
                remote = re.search(r"\bcluster_(st\w+|map)\s*\(|shared::cluster", body)
                if not remote:
                    continue
                seen += 1
                barrier = re.search(r"\bcluster_(sync|wait)\s*\(", body)
                assert barrier and barrier.start() < remote.start(), f"{name}: {kernel}"
    assert seen >= 1  # k_pair_stats
