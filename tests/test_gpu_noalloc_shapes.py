"""sw_search_pairs_noalloc at the edges of its kernel's shapes: 4 to 32 rows per
lane, one and several passes of 1,024 rows, ring blocks of 256 columns, more
subjects than one block item takes, and unsorted lengths; bit-exact against the
oracle."""
import numpy as np
import pytest

from helpers import oracle_all, seqset
from paper_2309_09609_gb300 import build as nvbuild
from paper_2309_09609_gb300 import swgb

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gaps", [(10, 2), (100000, 3)])
@pytest.mark.parametrize("subjects", [1, 83])
def test_edges(gaps, subjects):
    torch = pytest.importorskip("torch")
    nvbuild.build()
    rng = np.random.default_rng(subjects)
    lens = ([255, 0, 257, 256, 1, 4096, 225, 513] + list(rng.integers(0, 700, size=subjects)))
    db = seqset(rng, lens[:subjects] if subjects < 8 else lens, alpha=24)
    q = seqset(rng, [1024, 0, 1, 128, 129, 384, 385, 640, 641, 896, 897, 1023, 1025, 2049, 1151, 32],
               alpha=24)

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()

    out = torch.full((len(q), len(db)), -7, dtype=torch.int32, device="cuda")
    swgb.search_pairs_noalloc(dev(q.res), dev(q.offs), dev(q.lens), dev(db.res), dev(db.offs),
                              dev(db.lens), out, *gaps)
    want = oracle_all(q, db, *gaps)
    got = out.cpu().numpy()
    assert (got == want).all(), np.argwhere(got != want)[:5]


def test_query_lengths_at_the_edges_of_odd_pairs_of_rows():
    torch = pytest.importorskip("torch")
    nvbuild.build()
    rng = np.random.default_rng(11)
    db = seqset(rng, [255, 300, 1, 33] + list(rng.integers(0, 500, size=60)), alpha=24)
    q = seqset(rng, [191, 192, 193, 319, 320, 321, 448, 449, 576, 577, 704, 705, 832, 833, 960, 961],
               alpha=24)

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a)).cuda()

    out = torch.full((len(q), len(db)), -7, dtype=torch.int32, device="cuda")
    swgb.search_pairs_noalloc(dev(q.res), dev(q.offs), dev(q.lens), dev(db.res), dev(db.offs),
                              dev(db.lens), out, 10, 2)
    assert (out.cpu().numpy() == oracle_all(q, db, 10, 2)).all()
