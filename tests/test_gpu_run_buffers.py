"""A captured run holds its buffers by value: when a call between two runs of the same steps
replaces one of them (the statistical regime's first use, or a step that needs more room),
the run is captured again, with the same totals; when none was, it is replayed."""
import pytest

from paper_1608_01125_gb300 import binding, synth

pytestmark = pytest.mark.gpu

TOTALS = ("count", "weighted", "hsum", "hxor")


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.fixture(scope="module")
def beams():
    wl = synth.tiny_headon(n=6000, seed=25)
    a, b = synth.beams(wl)
    return wl, binding.to_device(a), binding.to_device(b)


def test_run_after_first_use_of_statistical_regime(beams):
    wl, a, b = beams
    with binding.Collider(a, b, wl.dt, wl.kappa) as col:
        r0 = col.run(0, 2)
        assert r0["count"] > 0
        n = col.debug_captures()
        col.build(0)
        col.surrogate_pairs(0, 6)
        r1 = col.run(0, 2)
        assert col.debug_captures() == n + 1  # its candidate list was replaced
        r2 = col.run(0, 2)
        assert col.debug_captures() == n + 1  # a replay
    for k in TOTALS:
        assert r0[k] == r1[k] == r2[k], k


@pytest.mark.parametrize("precision", [binding.FP32_BAND, binding.FP64])
def test_run_after_a_step_that_grew_the_buffers(beams, precision):
    wl, a, b = beams
    with binding.Collider(a, b, wl.dt, wl.kappa, precision=precision) as col:
        ref = col.run(0, 1)
        sparse = next(k for k in range(12, 1, -1) if col.run(k, 1)["count"] > 0)
        few = col.run(sparse, 1)
        assert ref["count"] > 512 > 64 > few["count"]
        col.debug_shrink_buffers(512)
        n = col.debug_captures()
        assert col.run(sparse, 1)["count"] == few["count"] and col.debug_captures() == n + 1
        col.build(0)
        col.collide(0)
        assert col.stats()["count"] == ref["count"] and col.stats()["retries"] > 0
        r1 = col.run(sparse, 1)
        assert col.debug_captures() == n + 2
        r0 = col.run(0, 1)
        for k in TOTALS:
            assert r1[k] == few[k] and r0[k] == ref[k], k
