"""The autotuner times what its knobs act on.  Without the statistical regime they act on
nothing: the current ones stay.  With it, the leaf bucket (which says what a cloud is) stays,
the others are chosen by the seeded traversal, the pairs and their exact labels are the same,
and the cached choice serves contexts of the same level and bucket only."""
import json
import math

import numpy as np
import pytest

from paper_1608_01125_gb300 import binding, synth

pytestmark = pytest.mark.gpu

N, L, KAPPA, STEP = 20000, 10, 1e16, 16


@pytest.fixture(scope="module")
def draw():
    import __graft_entry__
    __graft_entry__.build()
    wl = synth.statistical_1e8(n=N, seed=6)
    a, b = (binding.to_device(q) for q in synth.beams(wl))
    return wl, a, b


def pairs(col):
    g = col.surrogate_pairs(STEP, L, labels=True)
    return g["n_pairs"], np.sort(g["label"]), np.bincount(g["cloud_of_a"]).size


def test_knobs_stay_where_nothing_uses_them(draw, tmp_path):
    wl, a, b = draw
    cache = str(tmp_path / "t.json")
    for knobs in ((8, 256, 2, 64), (1, 1024, 8, 8)):
        with binding.Collider(a, b, wl.dt, KAPPA) as col:
            col.set_tuning(*knobs)
            assert tuple(col.autotune([STEP]).values()) == knobs
            assert tuple(col.tuning().values()) == knobs
            with pytest.raises(binding.TrilensError):
                col.autotune([-1])
    with binding.Collider(a, b, wl.dt, KAPPA) as col:
        plain = col.autotune([STEP], cache)
    with binding.Collider(a, b, wl.dt, KAPPA) as col:
        col.set_tuning(8, 256, 2, 64)
        got = col.autotune([STEP], cache)  # cached, but the bucket stays
        assert got["leaf_bucket"] == 8 and got["stack_depth"] == plain["stack_depth"]


@pytest.mark.parametrize("bucket", [1, 8])
def test_clouds_stay_and_the_seeded_traversal_is_timed(draw, tmp_path, bucket):
    wl, a, b = draw
    cache = str(tmp_path / "t.json")
    with binding.Collider(a, b, wl.dt, KAPPA) as col:  # an entry of a context without the regime
        col.set_tuning(bucket, 512, 4, 16)
        col.autotune([STEP], cache)
    with binding.Collider(a, b, wl.dt, KAPPA) as col:
        col.set_tuning(bucket, 512, 4, 16)
        before = pairs(col)
        assert before[0] > 50 and before[1].sum() > 0
        col.surrogate_collect([STEP], L)
        n = col.surrogate_info()["samples"]
        col.phase_ms(reset=True)
        got = col.autotune([STEP, STEP + 1], cache)
        launches = col.phase_ms()[1]
        assert launches["emit"] > 2  # hierarchies of the regime, not the exact path's trees
        assert got["leaf_bucket"] == bucket and col.tuning() == got
        assert col.surrogate_info()["samples"] == n and col.yield_() == (0.0, 0.0)
        after = pairs(col)
    assert after[0] == before[0] and after[2] == before[2]
    assert math.isclose(after[1].sum(), before[1].sum(), rel_tol=1e-12)
    assert np.allclose(after[1], before[1], rtol=1e-12)
    entries = json.load(open(cache))
    assert len(entries) == 2 and entries[1]["key"].endswith(f"_L{L}_b{bucket}")
    with binding.Collider(a, b, wl.dt, KAPPA) as col:
        col.set_tuning(bucket, 512, 4, 16)
        col.surrogate_collect([STEP], L)
        assert col.autotune([STEP], cache) == got
