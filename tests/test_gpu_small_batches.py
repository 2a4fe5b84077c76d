"""A small batch's plan: dealing its queries to two-query streams is left out where
no deal could be the faster layout, so that the call does not wait for it; the
options that ask for two queries per word still get them."""
import numpy as np
import pytest

from helpers import oracle_all, seqset
from paper_2309_09609_gb300 import build as nvbuild
from paper_2309_09609_gb300 import swgb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("opts", [{}, {"two_query": 2, "two_query_long": 2}, {"two_query": 0},
                                  {"two_query": 2, "two_query_long": 0}])
@pytest.mark.parametrize("subjects", [4, 130, 3000])
def test_layouts_of_small_batches(opts, subjects):
    nvbuild.build()
    rng = np.random.default_rng(subjects)
    db = seqset(rng, ([1700, 0, 2, 31] + list(rng.integers(0, 120, size=subjects)))[:subjects],
                alpha=24)
    q = seqset(rng, [0, 1, 14, 24, 33, 64, 65, 90, 200, 517], alpha=24)
    p = swgb.Database.from_seqset(db).plan(len(q), q.total, **opts)
    for nq in (10, 2, 1):
        got = p.search(q.res[:q.lens[:nq].sum()], q.lens[:nq])
        assert (got == oracle_all(q.subset(np.arange(nq)), db)).all()
        st = p.stats()
        asked = opts.get("two_query") == 2 and nq > 1
        assert (st["inter2_items"] > 0) == (asked and subjects > 64)
        assert (st["pair2_items"] > 0) == (nq > 1 and opts.get("two_query_long") == 2)


@pytest.mark.parametrize("opts", [{"two_query": 2, "two_query_long": 2},
                                  {"two_query": 2, "two_query_long": 0}])
def test_two_kernels_side_by_side(opts):
    # overlap_kernels acts only where the long and the short subjects go to
    # kernels of their own, as these options make them
    nvbuild.build()
    rng = np.random.default_rng(7)
    db = seqset(rng, [4000, 2500, 1700] + list(rng.integers(0, 900, size=600)), alpha=24)
    q = seqset(rng, [2100, 1, 77, 500, 1030], alpha=24)
    p = swgb.Database.from_seqset(db).plan(len(q), q.total, overlap_kernels=1, **opts)
    want = oracle_all(q, db)
    for _ in range(4):
        assert (p.search(q.res, q.lens) == want).all()
        st = p.stats()
        assert st["kernels_launched"] >= 2 and st["inter2_items"] > 0
        assert (st["pair2_items"] > 0) == (opts["two_query_long"] == 2)
