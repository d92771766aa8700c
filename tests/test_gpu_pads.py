"""Boxes padded by energy (the exact path's half-widths amp E^xp): bit-exact hit sets
against the FP64 brute force where the pads matter most: energies from below threshold to
far above the peak of the cross-section, broad and unequal spectra, single values, photons
without energy, at several crossing angles, and a batch whose instances differ."""
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


def beams(n, crossing, ea, eb, seed, div=5e-3):
    s = synth.BeamSpec(n, (1.0, 1.0), 3.0, div, ("lognormal", 5.0, 0.5))
    wl = synth.Workload("x", s, s, crossing, C * 2 * 10.0, 10.0, 4, 1e16, seed)
    a, b = synth.beams(wl)
    rng = np.random.default_rng(seed)
    for beam, (mean, sd) in ((a, ea), (b, eb)):
        beam["E"] = np.exp(math.log(mean) + sd * rng.standard_normal(n))
    return a, b


SPECTRA = [((5.0, 0.0), (5.0, 0.0)), ((0.6, 0.1), (0.6, 0.1)), ((20.0, 2.0), (20.0, 2.0)),
           ((0.01, 0.5), (500.0, 0.5)), ((1e5, 1.0), (1e5, 1.0)), ((3.0, 3.0), (0.2, 0.3))]


@pytest.mark.parametrize("crossing", [0.0, 0.9, math.pi / 2, 2.2])
@pytest.mark.parametrize("ea,eb", SPECTRA)
def test_spectra_and_angles(ea, eb, crossing):
    a, b = beams(1500, crossing, ea, eb, 51)
    a["E"][:3] = 0.0
    found = 0
    for kappa in (1e16, 1e18, 1e22):
        with binding.Collider(a, b, 10.0, kappa) as col:
            for k in (1, 2):
                ref, r = oracle.bruteforce(a, b, k, 10.0, kappa, cap=1 << 22)
                h, st = col.step_hits(k)
                assert np.array_equal(pairs(h), pairs(ref))
                assert st["hsum"] == r["hsum"] and st["hxor"] == r["hxor"]
                found += len(ref)
    assert found > 0 or crossing > 2.0 or ea[0] < 1.0


def test_batch_of_unlike_spectra():
    inst = [beams(300 + 40 * q, 0.3 * q, *SPECTRA[q % len(SPECTRA)], 60 + q) for q in range(8)]
    kappa = 1e18
    A, B = ([binding.to_device(q[s]) for q in inst] for s in (0, 1))
    with binding.Batch(A, B, 10.0, kappa) as col:
        got = np.asarray(col.run(0, 4))
    for q, (a, b) in enumerate(inst):
        ref = sum(oracle.bruteforce(a, b, k, 10.0, kappa, cap=1 << 22)[1]["count"]
                  for k in range(4))
        assert got[q, 0] == ref, q
