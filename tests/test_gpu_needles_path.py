"""The cases of test_gpu_needles.py are told by needles in both precisions at the step where
the beams' centres meet (all but the one with few queries, whose tree is the other beam's),
and sparse or nearly parallel beams by their boxes."""
import numpy as np
import pytest

from paper_1608_01125_gb300 import binding, synth
from test_gpu_needles import CASES, DT, KAPPA, beams

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def needles(a, b, kappa=KAPPA, **kw):
    with binding.Collider(a, b, DT, kappa, **kw) as col:
        with pytest.raises(binding.TrilensError):
            col.debug_needles()  # no step built
        col.build(2)
        return col.debug_needles()


@pytest.mark.parametrize("case", [c for c in CASES if c != "few queries"] + ["far", "strays"])
@pytest.mark.parametrize("precision", [binding.FP32_BAND, binding.FP64])
def test_dense_cases_take_needles(case, precision):
    a, b = CASES[case]() if case in CASES else beams(3000, seed=79)
    if case == "far":
        for q in (a, b):
            q["px"], q["py"] = q["px"] + 3000.0, q["py"] - 5000.0
    if case == "strays":
        for q, s in ((a, 1.0), (b, -1.0)):
            q["dx"][:5], q["dy"][:5], q["dz"][:5] = np.sin(0.3), 0.0, s * np.cos(0.3)
    assert needles(a, b, precision=precision)


def test_boxes_elsewhere():
    assert not needles(*beams(300))  # few photons meet a photon's box
    assert not needles(*beams(3000, div=1e-4))  # travel across the axis below the pads
    a, _ = beams(3000)
    assert not needles(a, synth.beams(synth.tiny_headon(n=2000, seed=3))[0])  # same direction
