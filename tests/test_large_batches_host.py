"""The stream layout of a batch of tens of thousands of queries, on the CPU: each
query once and whole, streams as even as dealing longest first gives, and in a
time that grows with the batch and not with its square."""
import heapq
import time

import numpy as np
import pytest

from paper_2309_09609_gb300 import build as nvbuild
from paper_2309_09609_gb300 import swgb

N, PAIRS = 60_000, 30_000


@pytest.fixture(scope="module", autouse=True)
def built():
    nvbuild.build()
    swgb.lib()


def test_layout_of_many_queries():
    rng = np.random.default_rng(6)
    lens = rng.integers(0, 400, size=N).astype(np.int32)
    t = time.perf_counter()
    strips, pairs = swgb.query_streams(lens, 32, PAIRS)
    seconds = time.perf_counter() - t
    # 3.6e9 comparisons where each query looked through all streams: 3 s and more
    assert seconds < 1.0
    need = np.maximum(1, -(-lens // 32))
    seen = np.zeros(N, dtype=np.int64)
    for half in (0, 2):
        q = strips[:, half]
        assert (np.bincount(q[q >= 0], minlength=N)[q[q >= 0]] == need[q[q >= 0]]).all()
        seen += np.bincount(q[q >= 0], minlength=N)
    assert (seen == need).all()
    heap = [0] * (2 * PAIRS)
    for s in np.sort(need)[::-1].tolist():
        heapq.heapreplace(heap, heap[0] + s)
    assert pairs[:, 1].max() <= max(heap)
