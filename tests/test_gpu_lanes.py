"""The lane-group kernel (csrc/lane_kernel.cu) against the oracle, bit-exact:
query lengths at the edges of its shapes (8, 16 and 32 lanes of 4 to 32 rows,
one and several passes), an odd number of subjects, subjects around the
8-residue chunks and the 64- to 256-column ring blocks, an empty query and
empty subjects, scores that saturate 16 bits, and the three gap classes."""
import numpy as np
import pytest

from helpers import concat, from_text, oracle_all, seqset
from paper_2309_09609_gb300 import build as nvbuild
from paper_2309_09609_gb300 import swgb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    nvbuild.build()
    swgb.lib()


@pytest.mark.parametrize("gaps", [(10, 2), (11, 1), (6, 3)])
@pytest.mark.parametrize("subjects", [1, 37, 701])
def test_query_lengths_at_the_edges_of_the_shapes(gaps, subjects):
    rng = np.random.default_rng(subjects + gaps[0])
    edges = [7, 8, 9, 63, 64, 65, 127, 128, 129, 255, 256, 257, 511, 512, 513]
    lens = (edges + list(rng.integers(0, 900, size=subjects)))[:subjects]
    db = seqset(rng, lens, alpha=24)
    q = seqset(rng, [0, 1, 4, 31, 32, 33, 129, 255, 257, 448, 449, 512, 513, 897, 1023, 1024, 1025,
                     1152, 2047, 2049], alpha=24)
    want = oracle_all(q, db, *gaps)
    d = swgb.Database.from_seqset(db)
    batch = d.plan(len(q), q.total, two_query=0, two_query_long=0, long_cutoff=300)
    got = batch.search(q.res, q.lens, *gaps)
    assert (got == want).all(), np.argwhere(got != want)[:5]
    one = d.plan(1, 2100)
    for i in range(len(q)):          # alone: other shapes for the longest subjects
        got = one.search(q.seq(i), q.lens[i:i + 1], *gaps)[0]
        assert (got == want[i]).all(), (int(q.lens[i]), np.argwhere(got != want[i])[:5])


def test_saturated_pairs_in_one_and_in_several_passes():
    rng = np.random.default_rng(3)
    m = rng.integers(-8, 3, size=(24, 24)).astype(np.int8)
    np.fill_diagonal(m, 100)
    base = seqset(rng, [1500])
    db = concat(base, seqset(rng, list(rng.integers(1, 700, size=90))), base.subset([0]))
    q = concat(base, seqset(rng, [40, 1300]), from_text("A" * 420))
    want = oracle_all(q, db, 10, 2, m.astype(np.int32))
    assert want.max() > 32767
    p = swgb.Database.from_seqset(db).plan(len(q), q.total, two_query=0, two_query_long=0)
    assert (p.search(q.res, q.lens, 10, 2, m) == want).all()
    assert p.stats()["recomputed_pairs"] >= 2


@pytest.mark.parametrize("m", [1153, 1500, 1537, 2200, 2305, 2948, 3073, 4200])
def test_chains_that_end_in_passes_of_fewer_rows(m):
    rng = np.random.default_rng(m)
    db = seqset(rng, [3000, 1, 33, 64, 257, 900, 2999, 0, 31, 1500, 2048, 7, 1100], alpha=24)
    q = seqset(rng, [m], alpha=24)
    got = swgb.Database.from_seqset(db).plan(1, m).search(q.res, q.lens, 10, 2)
    assert (got == oracle_all(q, db, 10, 2)).all()


def test_query_lengths_at_the_edges_of_odd_pairs_of_rows():
    rng = np.random.default_rng(8)
    db = seqset(rng, list(rng.integers(0, 500, size=301)), alpha=24)
    q = seqset(rng, [47, 48, 49, 79, 80, 81, 111, 112, 113, 144, 176, 208, 239, 240, 241, 288, 289,
                     352, 416, 417, 480, 481, 576, 704, 705, 832, 960, 961], alpha=24)
    d = swgb.Database.from_seqset(db)
    got = d.plan(len(q), q.total, two_query=0, two_query_long=0).search(q.res, q.lens, 10, 2)
    assert (got == oracle_all(q, db, 10, 2)).all()
