"""The int32 recompute of saturated pairs (csrc/intra_kernel.cu): on a device that
has no room for its clusters (injected on the host), and with as many pairs as
make a block each faster than clusters that take them in turn."""
import numpy as np
import pytest

from helpers import concat, oracle_all, seqset
from paper_2309_09609_gb300 import build as nvbuild
from paper_2309_09609_gb300 import swgb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    nvbuild.build()
    swgb.lib()


def saturating(rng, length, copies):
    """A query, a database with `copies` of it among others, a matrix that makes
    each copy's score exceed 16 bits."""
    m = np.full((24, 24), -4, np.int8)
    np.fill_diagonal(m, 11)
    q = seqset(rng, [length])
    return q, concat(*[q] * copies, seqset(rng, list(rng.integers(0, 300, size=70)))), m


@pytest.mark.parametrize("rows", [8, 16])
def test_without_clusters_every_pair_is_recomputed_on_a_block(rows, monkeypatch):
    q, db, m = saturating(np.random.default_rng(1), 3000, 3)
    want = oracle_all(q, db, 10, 2, m.astype(np.int32))
    d = swgb.Database.from_seqset(db)
    kernels = []
    for fault in (None, "clusters"):
        if fault:
            monkeypatch.setenv("SWGB_FAULT", fault)
        p = d.plan(1, 3000, intra_rows=rows)
        assert (p.search(q.res, q.lens, 10, 2, m) == want).all()
        assert p.stats()["recomputed_pairs"] == 3
        kernels.append(p.stats()["kernels_launched"])
    assert kernels[1] == kernels[0] - 1


@pytest.mark.parametrize("pairs", [1, 9, 10, 36, 37])
def test_pairs_of_few_passes_do_not_wait_for_one_another(pairs):
    # 36 pairs on 9 clusters, four in turn, took 4.4 times as long as 37 on a
    # block each
    q, db, m = saturating(np.random.default_rng(pairs), 3100, pairs)
    want = oracle_all(q, db, 10, 2, m.astype(np.int32))
    p = swgb.Database.from_seqset(db).plan(1, 3100)
    ms = []
    for _ in range(5):
        assert (p.search(q.res, q.lens, 10, 2, m) == want).all()
        ms.append(p.stats()["recompute_ms"])
    assert p.stats()["recomputed_pairs"] == pairs
    lone, lq, lm = saturating(np.random.default_rng(0), 3100, 37)
    p = swgb.Database.from_seqset(lq).plan(1, 3100)
    alone = []
    for _ in range(5):
        p.search(lone.res, lone.lens, 10, 2, lm)
        alone.append(p.stats()["recompute_ms"])
    assert min(ms) < 1.5 * min(alone), (min(ms), min(alone))


@pytest.mark.parametrize("rows", [8, 16])
@pytest.mark.parametrize("lengths", [[4100, 3000, 9000, 0, 5000], [12000] + [3000] * 11])
def test_recompute_of_pairs_of_several_lengths(lengths, rows):
    # both sides of the rule, pairs of unequal length to one cluster
    rng = np.random.default_rng(len(lengths))
    m = np.full((24, 24), -4, np.int8)
    np.fill_diagonal(m, 11)
    q = seqset(rng, lengths)
    db = concat(q, seqset(rng, list(rng.integers(0, 200, size=64))))
    want = oracle_all(q, db, 10, 2, m.astype(np.int32))
    p = swgb.Database.from_seqset(db).plan(len(q), q.total, intra_rows=rows)
    assert (p.search(q.res, q.lens, 10, 2, m) == want).all()
    assert p.stats()["recomputed_pairs"] == sum(n > 0 for n in lengths)
