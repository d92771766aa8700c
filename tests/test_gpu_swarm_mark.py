"""The marks of trilens_swarm_mark against the FP64 decision of every pair, at the
edges of the kernel's tiles (threads, words of marks, slices of beam B) and for
inputs its FP32 test must leave to FP64: nearly parallel pairs, directions that are
not unit vectors, pairs placed on the limit."""
import math

import numpy as np
import pytest

from paper_1608_01125_gb300 import binding, synth

pytestmark = pytest.mark.gpu

C, MEC2, RE = 0.299792458, 0.51099895, 2.8179403262e-15


def _sigma(s):
    b = np.sqrt((s - 1.0) / s)
    return 0.5 * math.pi * RE * RE / s * (
        (3.0 - b ** 4) * np.log((1.0 + b) ** 2 * s) - 2.0 * b * (2.0 - b * b))


def _marks(a, b, ha, hb, dt, kappa, first, steps):
    rmax = 1e6 * math.sqrt(kappa * _sigma(np.linspace(1.5, 3.0, 400001)).max() * (1 + 1e-6) / math.pi)
    reach = (rmax + 0.8660254037844387 * (ha + hb)) * (1.0 + 1e-6) + 1e-9
    t0, t1 = first * dt, (first + steps) * dt
    P = lambda q: np.stack([q["p" + c] for c in "xyz"])  # noqa: E731
    D = lambda q: np.stack([q["d" + c] for c in "xyz"])  # noqa: E731
    p = P(a)[:, :, None] - P(b)[:, None, :]
    v = C * (D(a)[:, :, None] - D(b)[:, None, :])
    s = a["E"][:, None] * b["E"][None, :] * (1.0 - D(a).T @ D(b))
    vv = (v * v).sum(0)
    with np.errstate(invalid="ignore", divide="ignore"):
        t = np.clip(-(p * v).sum(0) / vv, t0, t1)
    q = p + t * v
    ok = (s > 2.0 * MEC2 * MEC2 * (1 - 1e-9)) & (vv > 0) & ((q * q).sum(0) <= reach * reach + 1e-9)
    return ok.any(1), ok.any(0)


@pytest.mark.parametrize("na,nb", [(1, 1), (31, 33), (257, 129), (256, 1024), (300, 4099)])
@pytest.mark.parametrize("case", ["plain", "parallel", "nonunit"])
def test_marks_equal_the_fp64_decision(na, nb, case):
    import __graft_entry__
    __graft_entry__.build()
    rng = np.random.default_rng(na * 10007 + nb)
    wl = synth.ip_headon(n_mp=max(na, nb), seed=3)
    a, b = synth.beams(wl)
    a = {k: v[:na].copy() for k, v in a.items()}
    b = {k: v[:nb].copy() for k, v in b.items()}
    a["E"] *= rng.uniform(0.05, 1.0, na)  # some pairs below threshold
    if case == "parallel":  # half of beam B flies with beam A, exactly or nearly
        h = nb // 2 + 1
        for c in "xyz":
            b["d" + c][:h] = a["d" + c][rng.integers(0, na, h)] + (c == "x") * rng.choice([0.0, 1e-9, 1e-3], h)
    if case == "nonunit":
        f = rng.choice([1.0, 1.0 + 1e-4, 2.5], nb)
        for c in "xyz":
            b["d" + c] *= f
    for cube, first, steps in ((0.0, 0, 64), (0.05, 2, 3), (0.5, 0, 1)):
        ma, mb = binding.swarm_mark(binding.to_device(a), binding.to_device(b), cube, cube, wl.dt,
                                    1e16, first, steps)
        ra, rb = _marks(a, b, cube, cube, wl.dt, 1e16, first, steps)
        assert np.array_equal(ma.cpu().numpy() != 0, ra), (cube, first, steps)
        assert np.array_equal(mb.cpu().numpy() != 0, rb), (cube, first, steps)
