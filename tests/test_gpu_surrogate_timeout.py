"""The statistical regime on a hierarchy whose build's bounded wait ran out: the call returns
TRILENS_ERR_TIMEOUT without following links that were never written, whether it is the
context's first build (nothing in the buffers yet) or a later one."""
import ctypes
import math

import numpy as np
import pytest

from paper_1608_01125_gb300 import binding, synth

pytestmark = pytest.mark.gpu

N, L = 20000, 8


@pytest.fixture(scope="module")
def draw():
    import __graft_entry__
    __graft_entry__.build()
    wl = synth.tiny_headon(n=N, seed=12)
    a, b = (binding.to_device(q) for q in synth.beams(wl))
    with binding.Collider(a, b, wl.dt, 1e15) as col:
        ref = col.surrogate_pairs(0, L, labels=True)
    assert ref["n_pairs"] > 10 and ref["label"].sum() > 0
    return wl, a, b, ref


def same(g, ref):
    assert g["n_pairs"] == ref["n_pairs"]
    assert math.isclose(g["label"].sum(), ref["label"].sum(), rel_tol=1e-12)
    assert np.array_equal(np.sort(g["st"]), np.sort(ref["st"]))


@pytest.mark.parametrize("first", [True, False])
def again(col, step):
    """The pairs of a step without another trilens_build."""
    sp = binding.SurPairs(0, 0, *[None] * 9, 0.0)
    rc = binding.lib().trilens_surrogate_pairs(col.ctx, step, L, 1e30, ctypes.byref(sp))
    return rc, sp.n_pairs


@pytest.mark.parametrize("first", [True, False])
def test_call_after_expired_wait_builds_again(draw, first):
    wl, a, b, ref = draw
    with binding.Collider(a, b, wl.dt, 1e15) as col:
        if not first:
            same(col.surrogate_pairs(0, L, labels=True), ref)
        col.build(1)
        want = again(col, 1)
        assert want[0] == binding.OK and want[1] > 10
    with binding.Collider(a, b, wl.dt, 1e15) as col:
        if not first:
            same(col.surrogate_pairs(0, L, labels=True), ref)
        col.debug_set_spin_limit(2000)
        col.debug_stall_sort(True)
        col.build(1)
        assert again(col, 1)[0] == binding.ERR_TIMEOUT
        col.debug_stall_sort(False)
        col.debug_set_spin_limit(1 << 22)
        assert again(col, 1) == want


@pytest.mark.parametrize("first", [True, False])
def test_expired_wait(draw, first):
    wl, a, b, ref = draw
    with binding.Collider(a, b, wl.dt, 1e15) as col:
        if not first:
            same(col.surrogate_pairs(0, L, labels=True), ref)
        col.debug_set_spin_limit(2000)
        col.debug_stall_sort(True)
        with pytest.raises(binding.TrilensError) as ei:
            col.surrogate_pairs(1, L, labels=True)
        assert ei.value.code == binding.ERR_TIMEOUT
        col.debug_stall_sort(False)
        col.debug_set_spin_limit(1 << 22)
        same(col.surrogate_pairs(0, L, labels=True), ref)
