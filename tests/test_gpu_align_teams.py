"""sw_align with each team size (16, 4 and 1 warps to a pair, by the number of
pairs in the call): the same alignments as the oracle's, over paths that run
32 columns and more along the diagonal and in gaps of both kinds."""
import numpy as np
import pytest

from helpers import seqset
import oracle
from paper_2309_09609_gb300 import build as nvbuild
from paper_2309_09609_gb300 import swgb, synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pairs", [9, 600, 2700])
@pytest.mark.parametrize("gaps", [(10, 2), (0, 1), (3, 0)])
def test_every_team_size(pairs, gaps):
    nvbuild.build()
    rng = np.random.default_rng(pairs)
    base = seqset(rng, [420]).seq(0)

    def related(gap_at, gap):   # mutated, with one stretch deleted
        s = synth.mutate(rng, base, 0.15)
        return np.delete(s, np.arange(gap_at, gap_at + gap))

    cut = [(50, 1), (100, 31), (200, 32), (120, 33), (260, 70), (30, 300)]
    seqs = [base] + [related(*c) for c in cut] + [seqset(rng, [n]).seq(0) for n in (1, 31, 33, 257)]
    ss = synth.SeqSet(np.concatenate(seqs), np.array([s.size for s in seqs], np.int32))
    want = {}
    pq, ps = rng.integers(0, len(seqs), size=pairs), rng.integers(0, len(seqs), size=pairs)
    got = swgb.Database.from_seqset(ss).align(ss.res, ss.lens, pq, ps, *gaps)
    for k, (a, b) in enumerate(zip(pq.tolist(), ps.tolist())):
        if (a, b) not in want:
            want[a, b] = oracle.align(seqs[a], seqs[b], *gaps)
        assert got[k] == want[a, b], (a, b)


@pytest.mark.parametrize("top", [6, 127])
def test_scores_below_and_above_16_bits(top):
    # with an entry of 127 a pair of 420 could exceed 32767, so the call stores
    # direction bits; with 6 it stores H
    nvbuild.build()
    rng = np.random.default_rng(top)
    m = rng.integers(-6, 3, size=(24, 24)).astype(np.int8)
    np.fill_diagonal(m, top)
    base = seqset(rng, [420]).seq(0)
    seqs = [base, np.delete(base, np.arange(100, 140)), np.delete(synth.mutate(rng, base, 0.2), [7]),
            seqset(rng, [300]).seq(0)]
    ss = synth.SeqSet(np.concatenate(seqs), np.array([s.size for s in seqs], np.int32))
    pq, ps = np.repeat(np.arange(4), 4), np.tile(np.arange(4), 4)
    for repeat, gaps in ((1, (9, 1)), (1, (0, 0)), (1, (40000, 3)), (40, (5, 0)), (160, (11, 1))):
        a, b = np.tile(pq, repeat), np.tile(ps, repeat)
        got = swgb.Database.from_seqset(ss).align(ss.res, ss.lens, a, b, *gaps, m)
        want = [oracle.align(seqs[q], seqs[s], *gaps, m.astype(np.int32)) for q, s in zip(pq, ps)]
        assert got == want * repeat


@pytest.mark.parametrize("n", [64_999, 65_000, 65_001, 66_000])
def test_subjects_around_the_longest_whose_steps_fit_16_bits(n):
    nvbuild.build()
    rng = np.random.default_rng(n)
    q = seqset(rng, [90])
    s = seqset(rng, [n]).seq(0).copy()
    s[n - 70:n - 10] = q.seq(0)[20:80]   # the best alignment ends near the last column
    ss = synth.SeqSet(s, np.array([n], np.int32))
    got = swgb.Database.from_seqset(ss).align(q.res, q.lens, [0], [0], 10, 2)
    assert got[0] == oracle.align(q.seq(0), s, 10, 2)
