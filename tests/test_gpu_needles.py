"""Photon pairs told at the time they pass each other (needles): bit-exact hit sets against
the FP64 brute force for beams that take that path (dense, and with divergences that carry
a photon many collision radii across its path in a step): closing along each axis, in a
turned frame, far from the origin, with photons far off the beam's direction, at the step's
ends, in FP64 mode and as one run."""
import math

import numpy as np
import pytest

import oracle
from paper_1608_01125_gb300 import binding, synth

pytestmark = pytest.mark.gpu

C = 0.299792458
DT, KAPPA = 20.0, 1e14


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def pairs(h):
    h = np.asarray(h, dtype=np.int64).reshape(-1, 2)
    return h[np.lexsort((h[:, 1], h[:, 0]))]


def turned(beam, axis, angle):
    k = np.asarray(axis, float) / np.linalg.norm(axis)
    K = np.array([[0, -k[2], k[1]], [k[2], 0, -k[0]], [-k[1], k[0], 0]])
    R = np.eye(3) + math.sin(angle) * K + (1 - math.cos(angle)) * K @ K
    out = dict(beam)
    for q in "pd":
        v = R @ np.stack([beam[q + c] for c in "xyz"])
        for i, c in enumerate("xyz"):
            out[q + c] = np.ascontiguousarray(v[i])
    return out


def beams(n, crossing=0.0, div=20e-3, seed=71, nb=None):
    s = synth.BeamSpec(n, (0.3, 0.3), 3.0, div, ("lognormal", 5.0, 0.5))
    t = synth.BeamSpec(nb or n, (0.3, 0.3), 3.0, div, ("lognormal", 3.0, 0.7))
    wl = synth.Workload("x", s, t, crossing, C * 2 * DT, DT, 4, KAPPA, seed)
    return synth.beams(wl)


CASES = {
    "z": lambda: beams(3000),
    "x": lambda: tuple(turned(q, (0, 1, 0), math.pi / 2) for q in beams(3000, seed=72)),
    "y": lambda: tuple(turned(q, (1, 0, 0), math.pi / 2) for q in beams(3000, seed=73)),
    "crossing": lambda: beams(3000, crossing=1.0, seed=74),
    "crossing turned": lambda: tuple(turned(q, (1, -2, 0.5), 0.9)
                                     for q in beams(3000, crossing=0.4, seed=75)),
    "wide": lambda: beams(3000, div=60e-3, seed=76),
    "unequal": lambda: beams(4000, nb=1033, seed=77),
    "few queries": lambda: beams(33, nb=4000, seed=78),
}


@pytest.mark.parametrize("case", list(CASES) + ["far", "strays"])
def test_hit_sets(case):
    a, b = CASES[case]() if case in CASES else beams(3000, seed=79)
    if case == "far":
        for q in (a, b):
            q["px"] = q["px"] + 3000.0
            q["py"] = q["py"] - 5000.0
    if case == "strays":
        for q, s in ((a, 1.0), (b, -1.0)):
            q["dx"][:5], q["dy"][:5], q["dz"][:5] = math.sin(0.3), 0.0, s * math.cos(0.3)
    found = 0
    with binding.Collider(a, b, DT, KAPPA) as c32, \
            binding.Collider(a, b, DT, KAPPA, precision=binding.FP64) as c64:
        for k in range(5):
            ref, r = oracle.bruteforce(a, b, k, DT, KAPPA, cap=1 << 22)
            for col in (c32, c64):
                h, st = col.step_hits(k)
                assert np.array_equal(pairs(h), pairs(ref)), k
                assert st["hsum"] == r["hsum"] and st["hxor"] == r["hxor"]
            found += len(ref)
        assert c32.run(0, 5)["count"] == found
    assert found > 0
