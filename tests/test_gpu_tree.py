"""The exact path's order, trees and descent (tl_tree.cu) against the FP64 oracle's
brute force, at the edges of its tiles (32 photons per group and leaf, 1024 per tile),
with either beam the smaller one, and for beams whose frame is turned: crossing at any
angle, parallel, without a common direction.  The bar is bit-exact hit sets."""
import math

import numpy as np
import pytest

import oracle
from paper_1608_01125_gb300 import binding, synth

pytestmark = pytest.mark.gpu

C = 0.299792458


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def pairs(h):
    h = np.asarray(h, dtype=np.int64).reshape(-1, 2)
    return h[np.lexsort((h[:, 1], h[:, 0]))]


def turned(beam, axis, angle):
    """The beam turned about an axis through the origin."""
    k = np.asarray(axis, float) / np.linalg.norm(axis)
    K = np.array([[0, -k[2], k[1]], [k[2], 0, -k[0]], [-k[1], k[0], 0]])
    R = np.eye(3) + math.sin(angle) * K + (1 - math.cos(angle)) * K @ K
    out = dict(beam)
    for q in "pd":
        v = R @ np.stack([beam[q + c] for c in "xyz"])
        for i, c in enumerate("xyz"):
            out[q + c] = np.ascontiguousarray(v[i])
    return out


def check(a, b, dt, kappa, steps=(0, 1)):
    found = 0
    with binding.Collider(a, b, dt, kappa) as c32, \
            binding.Collider(a, b, dt, kappa, precision=binding.FP64) as c64:
        for k in steps:
            ref, r = oracle.bruteforce(a, b, k, dt, kappa, cap=1 << 21)
            for col in (c32, c64):
                h, st = col.step_hits(k)
                assert np.array_equal(pairs(h), pairs(ref)), k
                assert st["hsum"] == r["hsum"] and st["hxor"] == r["hxor"]
            found += len(ref)
    return found


@pytest.mark.parametrize("na,nb", [(1, 1), (1, 33), (31, 32), (33, 31), (1023, 1024), (1025, 1025),
                                   (33000, 40), (40, 33000), (5000, 32769)])
def test_sizes_at_tile_edges(na, nb):
    a, _ = synth.beams(synth.tiny_headon(n=na, seed=31))
    _, b = synth.beams(synth.tiny_headon(n=nb, seed=32))
    check(a, b, 10.0, min(1e18, 1e19 / min(na, nb)))


@pytest.mark.parametrize("crossing", [0.0, 0.02, 0.5, math.pi / 2, 2.5, math.pi - 0.05, math.pi])
@pytest.mark.parametrize("turn", [0.0, 0.7])
def test_crossing_angles_and_turned_beams(crossing, turn):
    s = synth.BeamSpec(1500, (1.0, 1.0), 3.0, 5e-3, ("lognormal", 5.0, 0.5))
    wl = synth.Workload("x", s, s, crossing, C * 2 * 10.0, 10.0, 4, 3e16, 33)
    a, b = (turned(q, (1.0, 2.0, -0.5), turn) for q in synth.beams(wl))
    n = check(a, b, 10.0, 3e16, (1, 2))
    assert n > 0 or crossing > 2.4  # nearly parallel photons stay below threshold


def test_no_common_direction_and_far_from_the_origin():
    rng = np.random.default_rng(34)
    a, b = synth.beams(synth.tiny_headon(n=1200, seed=35))
    for beam in (a, b):
        v = rng.standard_normal((3, 1200))
        v /= np.linalg.norm(v, axis=0)
        for i, c in enumerate("xyz"):
            beam["d" + c] = np.ascontiguousarray(v[i])
            beam["p" + c] = beam["p" + c] + 3e4
    assert check(a, b, 10.0, 1e17) > 0


def test_batch_of_mixed_sizes_and_angles():
    sizes = [(1, 5), (40, 33), (1024, 1500), (700, 0), (2049, 31)]
    A, B = [], []
    for q, (na, nb) in enumerate(sizes):
        s = synth.BeamSpec(max(na, nb), (0.7, 0.7), 3.0, 5e-3, ("lognormal", 5.0, 0.5))
        a, b = synth.beams(synth.Workload("x", s, s, 0.4 * q, C * 10.0, 10.0, 2, 3e16, 40 + q))
        A.append({k: v[:na].copy() for k, v in a.items()})
        B.append({k: v[:nb].copy() for k, v in b.items()})
    with binding.Batch(A, B, 10.0, 3e17) as bt:
        y = bt.run(0, 3)
    for q in range(len(sizes)):
        n = sum(oracle.bruteforce(A[q], B[q], k, 10.0, 3e17, cap=1 << 20)[1]["count"]
                for k in range(3)) if min(sizes[q]) else 0
        assert y[q, 0] == n, q
    assert y[:, 0].sum() > 100
