"""Plans of large capacity: one that no memory holds is refused with SW_ENOMEM
(in a process of its own: an exception that left the C ABI would end it), and a
batch that fills a large one is scored like any other."""
import subprocess
import sys
import textwrap

import numpy as np
import pytest

from helpers import oracle_all, seqset
from paper_2309_09609_gb300 import build as nvbuild
from paper_2309_09609_gb300 import swgb

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    nvbuild.build()
    swgb.lib()


@pytest.mark.parametrize("residues", [1 << 50, 1 << 59, (1 << 63) - 1])
def test_capacity_that_no_memory_holds_is_refused(residues):
    code = textwrap.dedent(f"""
        import numpy as np
        from paper_2309_09609_gb300 import swgb
        d = swgb.Database(np.arange(20, dtype=np.uint8), np.array([20], np.int32))
        try:
            d.plan(1, {residues})
        except swgb.SwError as e:
            assert e.status == swgb.SW_ENOMEM, e
            q = np.arange(20, dtype=np.uint8)
            print("refused", int(d.search(q, np.array([20], np.int32))[0, 0]))
        """)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.startswith("refused"), (r.returncode, r.stderr[-300:])


@pytest.mark.parametrize("n", [4095, 4097])
def test_batches_around_the_limit_of_two_segments_per_query(n):
    rng = np.random.default_rng(n)
    q = seqset(rng, rng.integers(0, 60, size=n), alpha=24)
    db = seqset(rng, [700, 1, 0, 33] + list(rng.integers(0, 90, size=30)), alpha=24)
    p = swgb.Database.from_seqset(db).plan(n, q.total, two_query=0, two_query_long=0)
    assert (p.search(q.res, q.lens) == oracle_all(q, db)).all()
