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
@pytest.mark.parametrize("gaps", [(10, 2), (0, 1)])
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
