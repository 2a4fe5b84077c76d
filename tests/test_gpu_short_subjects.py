"""Subjects of a few tens of residues, many of them (csrc/inter_kernel.cu): scores
against the oracle at the edges of its 32-row strips and 8-column chunks, and a
rate that does not fall with the subjects' length."""
import numpy as np
import pytest

from helpers import concat, oracle_all, seqset
from paper_2309_09609_gb300 import build as nvbuild
from paper_2309_09609_gb300 import swgb, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    nvbuild.build()
    swgb.lib()


def test_many_short_subjects_cost_as_much_per_residue_as_longer_ones():
    # a lane group's ramp of 32 steps is three times such a subject's columns:
    # 3.9 times the time of the longer subjects, where one query needs 1.2
    rng = np.random.default_rng(1)
    q = seqset(rng, [3000])
    ms = []
    for lens in (rng.integers(5, 16, 570_000), rng.integers(250, 351, 19_000)):
        p = swgb.Database.from_seqset(seqset(rng, lens)).plan(1, 3000)
        best = 1e9
        for _ in range(5):
            p.search(q.res, q.lens)
            best = min(best, p.stats()["search_ms"])
        ms.append(best)
    assert ms[0] < 2.2 * ms[1], ms


def test_two_query_streams_of_few_strips():
    # where most strips are a stream's first, whose border all warps fetched from
    # one word of L2: 3 times the time of the other layouts; and the same scores
    rng = np.random.default_rng(2)
    q, db = seqset(rng, [91] * 75), seqset(rng, [35] * 2071)
    d = swgb.Database.from_seqset(db)
    want = oracle_all(q, db)
    ms = []
    for two_query in (0, 2):
        p = d.plan(75, q.total, two_query=two_query)
        best = 1e9
        for _ in range(9):
            assert (p.search(q.res, q.lens) == want).all()
            best = min(best, p.stats()["search_ms"])
        ms.append(best)
    assert ms[1] < 2 * ms[0], ms


@pytest.mark.parametrize("gaps", [(10, 2), (11, 1), (6, 3)])
def test_scores_at_the_edges_of_strips_and_chunks(gaps):
    rng = np.random.default_rng(gaps[0])
    edges = [0, 1, 7, 8, 9, 15, 16, 17, 63, 64, 65]
    db = seqset(rng, edges + list(rng.integers(0, 30, 70_005)) + [1600, 2400], alpha=24)
    d = swgb.Database.from_seqset(db)
    lens = [1057, 1056, 1024, 1, 0, 31, 32, 33, 992]
    q = seqset(rng, lens, alpha=24)
    want = oracle_all(q, db, *gaps)
    for opts in ({}, {"two_query": 0, "overlap_kernels": 1}, {"use_graph": 0}):
        got = d.plan(len(q), q.total, **opts).search(q.res, q.lens, *gaps)
        assert (got == want).all(), (opts, np.argwhere(got != want)[:5])
    one = d.plan(1, 1100)
    for i in (0, 2, 8):
        got = one.search(q.seq(i), q.lens[i:i + 1], *gaps)
        assert (got[0] == want[i]).all(), lens[i]


def test_pairs_that_saturate_beside_many_short_subjects():
    rng = np.random.default_rng(4)
    m = rng.integers(-8, 3, size=(24, 24)).astype(np.int8)
    np.fill_diagonal(m, 127)
    q = seqset(rng, [280] * 8)
    hits = synth.SeqSet(np.concatenate([q.seq(i)[9:271] for i in (0, 3)]), np.array([262, 262]))
    db = concat(hits, seqset(rng, list(rng.integers(0, 13, 200_000))))
    want = oracle_all(q, db, 10, 2, m.astype(np.int32))
    assert (want > 32767).sum() == 2
    d = swgb.Database.from_seqset(db)
    for capacity in (0, 1):   # one listed pair, then a second round
        p = d.plan(8, q.total, flag_capacity=capacity)
        for _ in range(2):
            assert (p.search(q.res, q.lens, 10, 2, m) == want).all()
        assert p.stats()["recomputed_pairs"] >= 1 and p.stats()["overflow_rounds"] == capacity
