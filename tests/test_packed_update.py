"""The packed kernels' 16-bit cell update, restated on the CPU.

``model`` follows packed_cell of csrc/device_common.cuh step by step with 16-bit
wraparound: E floored at 0 (which stands for the zero term of Eq. 1), borders
of zeros, and S taken from the diagonal term x instead of H.  Against the
oracle it must give every score below the recompute threshold 32767 - max(SM)
- Go exactly, and flag every pair whose score reaches it, including pairs that
overflow 16 bits.
"""
import numpy as np
import pytest

import oracle


def wrap16(x):
    return ((x + 32768) & 0xFFFF) - 32768


def model(q, d, gap_open, gap_extend, sm):
    """S of each pair (q[k], d[k]); all queries of one length, all subjects too."""
    go, ge = gap_open + gap_extend, gap_extend
    n = d.shape[1]
    h_up, f = np.zeros((len(q), n + 1), np.int64), np.zeros((len(q), n), np.int64)
    s = np.zeros(len(q), np.int64)
    for i in range(q.shape[1]):
        w = sm[q[:, i][:, None], d].astype(np.int64)
        h_row, e = np.zeros_like(h_up), np.zeros(len(q), np.int64)
        for j in range(n):
            x = wrap16(h_up[:, j] + w[:, j])
            s = np.maximum(s, x)
            h = np.maximum(np.maximum(x, e), f[:, j])
            t = wrap16(h - go)
            e = np.maximum(np.maximum(wrap16(e - ge), t), 0)
            f[:, j] = np.maximum(wrap16(f[:, j] - ge), t)
            h_row[:, j + 1] = h
        h_up = h_row
    return s


@pytest.mark.parametrize("top,gaps", [(11, (10, 2)), (11, (11, 1)), (11, (0, 0)), (11, (0, 1)),
                                      (11, (8000, 8000)), (127, (10, 2)), (127, (0, 1))])
def test_scores_and_flags(top, gaps):
    rng = np.random.default_rng(top + gaps[0])
    sm = rng.integers(-6, 3, size=(24, 24)).astype(np.int8)
    np.fill_diagonal(sm, top)
    m, n = (275, 290) if top == 127 else (60, 70)
    q = rng.integers(0, 20, size=(8, m))
    d = rng.integers(0, 20, size=(8, n))
    for k in range(6):   # related pairs: identical stretches, some with a gap in them
        keep = m - 3 * k
        d[k, 5:5 + keep] = q[k, :keep]
        if k % 2:
            d[k, 100 % n:] = np.roll(d[k, 100 % n:], 3)
    want = np.array([oracle.search([a.astype(np.uint8)], [b.astype(np.uint8)], *gaps, sm)[0, 0]
                     for a, b in zip(q, d)])
    got = model(q, d, *gaps, sm)
    threshold = 32767 - int(sm.max()) - (gaps[0] + gaps[1])
    assert ((got >= threshold) == (want >= threshold)).all()
    assert (got[want < threshold] == want[want < threshold]).all()
    if top == 127 and gaps == (10, 2):
        assert (want > 32767).any()      # pairs that overflow 16 bits are among them
