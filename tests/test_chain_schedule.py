"""The stage schedule of a chain (lane_chain in csrc/lane_kernel.cu): the passes
of a subject pair on the warps of a block, with a barrier every 64 steps.

Restated here: every border column is written in an earlier stage than the
one that reads it (the next pass reads a stage's columns within that stage), it
is read before the warp's next pass overwrites it, a warp's passes do not
overlap, and every warp meets the same number of barriers.  Passes of 4 rows per
lane write a column 31 steps after reading it, the others 63 (`skews`).
"""
import itertools

import pytest

W, LAG, STAGE = 4, 2, 64


@pytest.mark.parametrize("passes", [2, 3, 4, 5, 8, 9, 26])
@pytest.mark.parametrize("n", [1, 30, 33, 64, 97, 200, 417, 449, 513, 2000])
def test_borders_are_written_before_and_read_before_overwritten(passes, n):
    spass = (n + 63 + STAGE - 1) // STAGE
    period = max(spass, W * LAG)
    start = [p // W * period + p % W * LAG for p in range(passes)]
    end = start[-1] + spass
    # every pass but the last has one number of rows, the last may have fewer
    for skews in itertools.product((31, 63), (31, 63)):
        skew = [skews[0]] * (passes - 1) + [skews[1]]
        for p in range(1, passes):
            for j in range(n):
                read = start[p] + j // STAGE
                assert start[p - 1] + (j + skew[p - 1]) // STAGE < read
                if p - 1 + W < passes:
                    assert read < start[p - 1 + W] + (j + skew[p - 1 + W]) // STAGE
        for p in range(passes):
            assert (n + skew[p] + STAGE - 1) // STAGE <= spass
    for p in range(passes):
        assert start[p] + spass <= end
        if p + W < passes:
            assert start[p] + spass <= start[p + W]
