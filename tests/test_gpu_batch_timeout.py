"""A batch whose cell scan's bounded wait runs out (a tile that never publishes) returns
TRILENS_ERR_TIMEOUT, in a captured run and step by step, and the context works on: its
instances are large enough for trees of three and more levels, whose upper ones must not be
built over sums that are not valid."""
import numpy as np
import pytest

from paper_1608_01125_gb300 import binding, synth

pytestmark = pytest.mark.gpu

SIZES = ((40000, 36000), (33000, 50001), (2000, 41000), (35000, 900))
DT, KAPPA = 10.0, 1e14


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def test_expired_wait_of_a_batch():
    a = [synth.beams(synth.tiny_headon(n=na, seed=40 + q))[0] for q, (na, _) in enumerate(SIZES)]
    b = [synth.beams(synth.tiny_headon(n=nb, seed=50 + q))[1] for q, (_, nb) in enumerate(SIZES)]
    ref = []
    for q in range(len(SIZES)):
        with binding.Collider(a[q], b[q], DT, KAPPA) as col:
            r = col.run(0, 2)
            ref.append([r["count"], r["weighted"]])
    assert all(r[0] > 0 for r in ref)
    with binding.Batch(a, b, DT, KAPPA) as col:
        for rep in range(2):
            col.debug_set_spin_limit(2000)
            col.debug_stall_sort(True)
            with pytest.raises(binding.TrilensError) as ei:
                col.run(0, 2)
            assert ei.value.code == binding.ERR_TIMEOUT
            col.build(0)
            with pytest.raises(binding.TrilensError) as ei:
                col.collide(0)
            assert ei.value.code == binding.ERR_TIMEOUT
            col.debug_stall_sort(False)
            col.debug_set_spin_limit(1 << 22)
            y = col.run(0, 2)
            assert np.array_equal(y, np.array(ref)), rep
            col.build(0)
            col.collide(0)
            one = col.stats()["count"]
            assert 0 < one <= sum(r[0] for r in ref)
