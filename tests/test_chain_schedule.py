"""The stage schedule of a chain (lane_chain in csrc/lane_kernel.cuh): the
passes of a subject pair on the warps of a block, with a barrier every 32 steps.

Restated here: every border column is written in an earlier stage than the one
that fetches it (stage k fetches the columns of stage k + 1, the first also its
own), it is read before the warp's next pass overwrites it, a warp's passes do
not overlap, and every warp meets the same number of barriers.  Passes of 4 rows
per lane write a column 31 steps after reading it, the others 63 (`skew`).
"""
import pytest

W, STAGE = 4, 32


@pytest.mark.parametrize("passes", [2, 3, 4, 5, 8, 9, 26])
@pytest.mark.parametrize("n", [1, 30, 33, 64, 97, 200, 417, 449, 513, 2000])
@pytest.mark.parametrize("full,last,tail", [(4, 4, 1), (8, 4, 1), (8, 8, 1), (16, 4, 1), (16, 16, 1),
                                            (8, 4, 3), (16, 8, 4), (16, 4, 2)])
def test_borders_are_written_before_and_read_before_overwritten(passes, n, full, last, tail):
    rows = [full] * (passes - tail) + [last] * tail
    if len(rows) > passes:
        return
    lag = 3 if full == 4 else 4

    def stages(pr):
        return (n + (31 if pr == 4 else 63) + STAGE - 1) // STAGE

    spass = stages(full)
    period = max(spass, W * lag)
    start = [p // W * period + p % W * lag for p in range(passes)]
    end = start[-1] + spass
    skew = [31 if pr == 4 else 63 for pr in rows]
    for p in range(1, passes):
        for j in range(n):
            read = start[p] + max(j // STAGE - 1, 0)
            assert start[p - 1] + (j + skew[p - 1]) // STAGE < read
            if p - 1 + W < passes:
                assert read < start[p - 1 + W] + (j + skew[p - 1 + W]) // STAGE
    for p in range(passes):
        own = stages(rows[p])
        assert own <= spass and start[p] + own <= end
        if p + W < passes:
            assert start[p] + spass <= start[p + W]


@pytest.mark.parametrize("passes", [2, 105, 128, 129, 140])
@pytest.mark.parametrize("n", [1, 33, 400, 12_500])
def test_recompute_over_a_cluster(passes, n):
    """recompute_kernel (csrc/intra_kernel.cu): the stages of 32 steps of the
    block recompute over the 128 warps of a cluster; a stage's reads fetch the
    next one's 32 columns."""
    warps, lag = 128, 3
    spass = (n + 31 + 31) // 32
    period = max(spass, lag * warps)
    start = [p // warps * period + p % warps * lag for p in range(passes)]
    for p in range(1, passes):
        for j in range(0, n, 7):
            read = start[p] + (0 if j < 32 else j // 32 - 1)
            assert start[p - 1] + (j + 31) // 32 < read
            if p - 1 + warps < passes:
                assert read < start[p - 1 + warps] + (j + 31) // 32
    assert all(start[p] + spass <= start[p + warps] for p in range(passes - warps))


@pytest.mark.parametrize("warps", [1, 4, 16])
@pytest.mark.parametrize("passes", [2, 5, 17, 40])
@pytest.mark.parametrize("n", [1, 15, 17, 47, 300, 1111])
def test_alignment_teams(warps, passes, n):
    """align_forward (csrc/align_kernel.cu): stages of 16 steps, a stage's reads
    fetch the next one's 16 columns."""
    stage, lag = 16, 4
    spass = (n + 31 + stage - 1) // stage
    period = max(spass, lag * warps)
    start = [p // warps * period + p % warps * lag for p in range(passes)]
    for p in range(1, passes):
        for j in range(n):
            read = start[p] + (0 if j < stage else j // stage - 1)
            assert start[p - 1] + (j + 31) // stage < read
            if p - 1 + warps < passes:
                assert read < start[p - 1 + warps] + (j + 31) // stage
    assert all(start[p] + spass <= start[p + warps] for p in range(passes - warps))


@pytest.mark.parametrize("passes", [2, 4, 5, 9, 17])
@pytest.mark.parametrize("n", [1, 33, 250, 353, 417, 1025, 1100])
def test_caller_memory_chains(passes, n):
    """na_chain (csrc/noalloc.cu): borders through rings of 256 columns between
    neighbouring warps, through a whole row from the last warp to the first."""
    ring, STAGE, LAG = 256, 64, 2
    spass = (n + 31 + STAGE - 1) // STAGE
    period = max(spass + LAG, W * LAG)
    start = [p // W * period + p % W * LAG for p in range(passes)]

    def write(p, j):
        return start[p] + (j + 31) // STAGE

    for p in range(1, passes):
        for j in range(n):
            read = start[p] + j // STAGE
            assert write(p - 1, j) < read
            overwrites = [write(p - 1 + W, j)] if p - 1 + W < passes else []
            if p % W:                                    # a ring: the same slot, later columns
                overwrites += [write(p - 1, k) for k in range(j + ring, n, ring)]
                if p - 1 + W < passes:
                    overwrites += [write(p - 1 + W, k) for k in range(j % ring, n, ring)]
            assert all(read < o for o in overwrites)
    assert all(start[p] + spass <= start[p + W] for p in range(passes - W))
