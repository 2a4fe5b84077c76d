"""sw_align's buffers: calls whose inputs or results are too large for the pinned
memory that the database keeps, calls that find too little device memory to keep H
of every cell, and device memory kept for later calls given back to a plan."""
import numpy as np
import pytest

from helpers import seqset
import oracle
from paper_2309_09609_gb300 import build as nvbuild
from paper_2309_09609_gb300 import swgb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    nvbuild.build()
    swgb.lib()


@pytest.mark.parametrize("queries,long", [(10, 0), (42_000, 0), (10, 600), (42_000, 600)])
def test_inputs_and_results_beyond_the_pinned_memory(queries, long):
    # 16 MiB: 42,000 queries of 400 go up beyond it, 600 slots of 35,400 come back
    rng = np.random.default_rng(queries + long)
    q = seqset(rng, [400] * queries)
    s = seqset(rng, [35_000, 90, 0, 300])
    d = swgb.Database.from_seqset(s)
    pq = np.concatenate([np.arange(10), np.full(long, 3)])
    ps = np.concatenate([np.arange(10) % 4, np.zeros(long, int)])
    want = {}
    for _ in range(2):
        got = d.align(q.res, q.lens, pq, ps)
        for a, b, g in zip(pq.tolist(), ps.tolist(), got):
            if (a, b) not in want:
                want[a, b] = oracle.align(q.seq(a), s.seq(b), 10, 2)
            assert g == want[a, b], (a, b)


def leave_free(torch, nbytes):
    """Takes device memory until about nbytes are free; returns what holds it."""
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free = torch.cuda.mem_get_info()[0]
    return torch.empty(free - nbytes, dtype=torch.uint8, device="cuda")


def test_direction_bits_where_memory_for_h_is_short():
    # H of these cells takes 618 MiB, their bits 155
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(5)
    q = seqset(rng, [2900] * 3)
    s = seqset(rng, [35_000] * 3)
    d = swgb.Database.from_seqset(s)
    args = (q.res, q.lens, [0, 1, 2], [2, 0, 1])
    want = d.align(*args)
    d.align(*args, 40_000, 3)                # penalties beyond 16 bits: bits, and their kernel loaded
    held = leave_free(torch, 400 << 20)
    try:
        got = d.align(*args)
    finally:
        del held
        torch.cuda.empty_cache()
    assert got == want


def test_memory_kept_for_alignments_gives_way_to_a_plan_and_a_search():
    # the two pairs' 412 MiB stay with the database; a plan, then a host-order
    # scores buffer, finds 200 MiB less than it needs outside of them
    torch = pytest.importorskip("torch")
    rng = np.random.default_rng(6)
    q = seqset(rng, [2900] * 2)
    s = seqset(rng, [35_000] * 2 + [40] * 70_000)
    d = swgb.Database.from_seqset(s)

    def used_by(make):
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        kept = make()
        return before - torch.cuda.mem_get_info()[0], kept

    need, plan = used_by(lambda: d.plan(1200, 20_000))
    scores, want = used_by(lambda: plan.search(q.res[:90], np.array([90], np.int32)))
    assert scores > 300 << 20
    plan.close()
    pairs = (q.res, q.lens, [0, 1], [1, 0])
    aligned = d.align(*pairs)
    for extra in (-(200 << 20), scores - (200 << 20)):
        d.align(*pairs)
        held = leave_free(torch, need + extra)
        try:
            plan = d.plan(1200, 20_000)
            if extra > 0:
                assert (plan.search(q.res[:90], np.array([90], np.int32)) == want).all()
        finally:
            del held
            torch.cuda.empty_cache()
        plan.close()
    assert d.align(*pairs) == aligned
