"""Marks where many warps find the same macro-photons at the same time: every warp of a block
adds to the same words of marks, which the others read to skip what is found.  Dense swarms
mark everything, sparse ones a part; the marks are those of the FP64 decision, every time."""
import numpy as np
import pytest

from paper_1608_01125_gb300 import binding, synth
from test_gpu_swarm_mark import _marks

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cube,steps", [(3.0, 64), (0.3, 4), (0.1, 64)])
def test_marks_do_not_depend_on_the_warps_order(cube, steps):
    import __graft_entry__
    __graft_entry__.build()
    wl = synth.ip_headon(n_mp=2000, seed=17)
    a, b = synth.beams(wl)
    a = {k: v[:1999].copy() for k, v in a.items()}
    ra, rb = _marks(a, b, cube, cube, wl.dt, 1e15, 0, steps)
    assert ra.any() and rb.any()
    da, db = binding.to_device(a), binding.to_device(b)
    for _ in range(20):
        ma, mb = binding.swarm_mark(da, db, cube, cube, wl.dt, 1e15, 0, steps)
        assert np.array_equal(ma.cpu().numpy() != 0, ra)
        assert np.array_equal(mb.cpu().numpy() != 0, rb)
