"""The seeded traversal of the statistical regime (exact labels of the level-L pairs, exact
fallback of a part of them) with every knob it has, in parts and with buffers it must grow:
deep and shallow stacks with their spill areas, work handed on at once, late or never, leaf
buckets of 1 to 32 photons.  The labels are the oracle's hits attributed to the pairs, the
fallback's yield is the sum of the labels of the pairs that fell back."""
import math

import numpy as np
import pytest

import oracle
from paper_1608_01125_gb300 import binding, synth

pytestmark = pytest.mark.gpu

N, L, KAPPA, STEP = 40000, 10, 3e15, 16


@pytest.fixture(scope="module")
def draw():
    import __graft_entry__
    __graft_entry__.build()
    wl = synth.statistical_1e8(n=N, seed=8)
    a, b = synth.beams(wl)
    hits, r = oracle.tree(a, b, STEP, wl.dt, KAPPA, nthreads=8, cap=1 << 22)
    assert len(hits) > 1000
    return wl, a, b, hits, r


def check(col, draw, tau=None):
    wl, a, b, hits, r = draw
    g = col.surrogate_pairs(STEP, L, tau=tau, labels=True)
    lab, outside = oracle.cloud_labels(a, b, hits, g["cloud_of_a"], g["cloud_of_b"], g["cloud"])
    assert outside == 0 and g["n_pairs"] > 50
    assert np.allclose(g["label"], lab, rtol=1e-12, atol=1e-12 * lab.max())
    assert math.isclose(g["label"].sum(), r["weighted"], rel_tol=1e-9)
    return g


KNOBS = [(1, 512, 4, 16), (8, 512, 4, 16), (32, 512, 4, 16), (4, 64, 4, 16), (4, 4096, 1, 16),
         (4, 128, 8, 16), (2, 64, 2, 2), (4, 64, 2, 5), (2, 64, 2, 0), (1, 64, 8, 1)]


@pytest.mark.parametrize("precision", [binding.FP32_BAND, binding.FP64])
@pytest.mark.parametrize("knobs", KNOBS)
def test_labels_with_every_knob(draw, knobs, precision):
    wl, a, b = draw[:3]
    with binding.Collider(a, b, wl.dt, KAPPA, precision=precision) as col:
        col.set_tuning(*knobs)
        check(col, draw)


@pytest.mark.parametrize("parts", [2, 5, 64])
def test_labels_in_parts(draw, parts):
    wl, a, b = draw[:3]
    with binding.Collider(a, b, wl.dt, KAPPA) as col:
        col.debug_set_parts(parts)
        check(col, draw)


@pytest.mark.parametrize("knobs", [(4, 512, 4, 16), (2, 64, 2, 2)])
@pytest.mark.parametrize("cap", [64, 1000])
def test_labels_with_buffers_that_grow(draw, knobs, cap):
    wl, a, b = draw[:3]
    with binding.Collider(a, b, wl.dt, KAPPA) as col:
        col.set_tuning(*knobs)
        check(col, draw)
        col.debug_shrink_buffers(cap)  # hits, band, leaf pairs, spill areas, queue
        check(col, draw)


@pytest.mark.parametrize("knobs", [(4, 512, 4, 16), (2, 64, 2, 2), (1, 64, 8, 0)])
def test_partial_fallback_with_knobs(draw, knobs):
    wl, a, b = draw[:3]
    with binding.Collider(a, b, wl.dt, KAPPA) as col:
        col.set_tuning(*knobs)
        col.surrogate_train([STEP - 1, STEP, STEP + 1], L, epochs=2, seed=3)
        g = check(col, draw, tau=1e30)
        spread = np.sqrt(np.exp(np.clip(g["net"][:, 1].astype(np.float64), -12, 12)))
        tau = float(np.quantile(spread, 0.6))
        for shrink in (False, True):
            if shrink:
                col.debug_shrink_buffers(64)
            g = check(col, draw, tau=tau)
            fb = g["fallback"].astype(bool)
            assert 0 < fb.sum() < len(fb) and g["label"][fb].sum() > 0
            assert math.isclose(g["fallback_exact"], g["label"][fb].sum(), rel_tol=1e-9)
            col.build(STEP)
            s = col.surrogate_step(STEP, L, tau)
            assert s["fallback_pairs"] == fb.sum()
            assert math.isclose(s["fallback_yield"], g["fallback_exact"], rel_tol=1e-9)
