"""The tuner times only options that choose code: an option that the library checks
and ignores would be tuned by the noise of repeats."""
import types

import pytest

from paper_2309_09609_gb300 import tune


def test_options_without_effect_are_not_timed():
    sp = tune.space(types.SimpleNamespace(max_length=35_000), 20)
    calls = []
    best, _ = tune.descend(tune.timed(sp), lambda o: calls.append(o) or float(len(calls)))
    assert best == {"two_query": 1, "long_cutoff": 1500, "intra_rows": 8}
    assert all(set(o) == {"two_query", "long_cutoff", "intra_rows"} for o in calls)


@pytest.mark.gpu
def test_tuned_options_hold_the_defaults_of_the_others():
    import numpy as np
    from helpers import seqset
    from paper_2309_09609_gb300 import build, swgb
    build.build()
    rng = np.random.default_rng(0)
    d = swgb.Database.from_seqset(seqset(rng, [2000] + [100] * 99))
    t = tune.tune(d, seqset(rng, [50, 400]), cache=None, repeats=1)
    assert set(t["options"]) == set(tune.space(d, 2))
    assert t["options"]["rows_per_thread"] == 32 and t["options"]["warps_per_block"] == 8
    assert all("rows_per_thread" not in o for o, _ in t["timings"])
