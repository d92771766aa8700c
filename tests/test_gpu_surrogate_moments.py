"""The clouds' moments from the running sums over the sorted photons, at the sizes where
their blocks (1024 photons), chunks (32) and thread groups (256) begin and end: every
listed pair's photon counts, weight sums, mean log-energies and mean directions against
plain float64 sums over the clouds' photons.

Tolerances: ln E is an FP32 logarithm (1 ulp of at most 4: 2.4e-7) of an FP32 energy
(6e-8), stored in FP32 (2.4e-7); directions are FP32 in and out (2 x 6e-8); logarithms of
counts and weight sums (below 16) are FP32 (1e-6)."""
import numpy as np
import pytest
import torch

from paper_1608_01125_gb300 import binding

pytestmark = pytest.mark.gpu


def _beam(n, sign, seed, weights):
    g = torch.Generator(device="cuda").manual_seed(seed)
    f = dict(dtype=torch.float64, device="cuda", generator=g)
    d = torch.randn((3, n), **f) * 0.05
    d[2] = sign
    d /= d.norm(dim=0)
    b = {k: torch.randn(n, **f) for k in ("px", "py", "pz")}
    b.update({k: d[i].contiguous() for i, k in enumerate(("dx", "dy", "dz"))})
    b["E"] = torch.exp(1.0 + 0.5 * torch.randn(n, **f)).clamp(0.1, 50.0)
    b["w"] = (1.0 + 9.0 * torch.rand(n, **f) if weights
              else torch.ones(n, dtype=torch.float64, device="cuda"))
    return b


@pytest.mark.parametrize("weights", [False, True])
@pytest.mark.parametrize("na,nb", [(1, 2), (31, 33), (32, 255), (256, 1), (1023, 1025),
                                   (1024, 2048), (2049, 65), (40001, 32768)])
def test_moments_of_the_clouds(na, nb, weights):
    import __graft_entry__
    __graft_entry__.build()
    a, b = _beam(na, 1.0, 3, weights), _beam(nb, -1.0, 4, weights)
    with binding.Collider(a, b, 5.0, 1e14) as col:
        for level in (3, 9):
            g = col.surrogate_pairs(0, level, labels=False)
            assert g["n_pairs"] > 0
            feat = g["feat"].astype(np.float64)
            for side, (beam, n) in enumerate(((a, na), (b, nb))):
                c = {k: v.cpu().numpy() for k, v in beam.items()}
                ids, at = np.unique(g["cloud_of_b" if side else "cloud_of_a"],
                                    return_inverse=True)

                def total(x):
                    return np.bincount(at, weights=x, minlength=len(ids))

                sw = total(c["w"])
                row = np.searchsorted(ids, g["cloud"][:, side])
                cols = {9 + side: np.log(total(np.ones(n))), 11 + side: np.log(sw)}
                for q, want in cols.items():
                    assert np.allclose(feat[:, q], want[row], rtol=0, atol=1e-6), (level, q)
                mle = total(c["w"] * np.log(c["E"])) / sw
                assert np.allclose(feat[:, 13 + side], mle[row], rtol=0, atol=6e-7), level
                for k, axis in enumerate("xyz"):
                    m = total(c["w"] * c["d" + axis]) / sw
                    assert np.allclose(feat[:, 17 + 3 * side + k], m[row], rtol=0,
                                       atol=1.5e-7), (level, axis)
