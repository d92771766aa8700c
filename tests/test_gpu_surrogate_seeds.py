"""What the network gains on beam shapes it was not trained on does not hang on the seed: for
each of several seeds (initial weights and order of the samples), a network trained on eight
shapes of the family of statistical workloads estimates twelve others' yields with a smaller
mean error than the ST rate alone and than that rate times the scale fitted in training.  A
seed stands for one training, whatever order the samples were collected in."""
import os
import struct

import numpy as np
import pytest

from paper_1608_01125_gb300 import binding, synth

pytestmark = pytest.mark.gpu

N, L = 1_000_000, 14
STEPS = list(range(6, 27))
TRAIN, FRESH = list(range(1, 9)), list(range(201, 213))


def collect(i):
    wl = synth.statistical_family(i, n=N)
    a, b = synth.beams(wl)
    with binding.Collider(a, b, wl.dt, wl.kappa) as col:
        col.surrogate_collect(STEPS, L)
        return col.surrogate_dataset()


def fitted(samples, seed, path):
    """Parameters, normalisation, scale of the calibrated network and of the baseline."""
    a, b = synth.beams(synth.statistical_family(1, n=1000))
    with binding.Collider(a, b, 20.0, 2e13) as col:
        for x, lab, st in samples:
            col.surrogate_add_samples(x, lab, st, L)
        col.surrogate_fit(epochs=30, seed=seed)
        info = col.surrogate_info()
        col.surrogate_save(path)
    blob = open(path, "rb").read()
    assert blob[:8] == b"TRLSUR03" and struct.unpack("<2i", blob[8:16])[1] == binding.MLP_PARAMS
    v = np.frombuffer(blob[-4 * (48 + binding.MLP_PARAMS):], np.float32)
    return v[48:].copy(), v[:48].copy(), info


def test_every_seed_beats_the_st_rate_on_fresh_shapes(tmp_path):
    import torch
    import __graft_entry__
    __graft_entry__.build()
    train = [collect(i) for i in TRAIN]
    fresh = [collect(i) for i in FRESH]
    path = str(tmp_path / "m.bin")

    def estimate(p, norm, info, x, st):
        dev = lambda v: torch.tensor(v, device="cuda")  # noqa: E731
        mu = binding.mlp_forward(dev(p), dev(norm), dev(x))[:, 0].double().cpu().numpy()
        base = np.float32(info["st_calib"]) * st.astype(np.float64) + 1.0
        return info["calib"] * float((base * np.exp(np.minimum(mu, 30.0))).sum())

    yields = np.array([lab.sum() for _, lab, _ in fresh])
    rate = np.array([st.astype(np.float64).sum() for _, _, st in fresh]) / yields - 1.0
    models = []
    for seed in (1, 2, 3, 4):
        p, norm, info = fitted(train, seed, path)
        models.append(p)
        net = np.array([estimate(p, norm, info, x, st) for x, _, st in fresh]) / yields - 1.0
        scaled = (1.0 + rate) * info["st_calib"] - 1.0
        m = [float(np.abs(v).mean()) for v in (net, rate, scaled)]
        print(f"seed {seed}: network {m[0]:.2%} (median {np.median(np.abs(net)):.2%}) "
              f"ST rate {m[1]:.2%} scaled {m[2]:.2%}")
        assert m[0] < m[1] and m[0] < m[2], seed
    assert not np.array_equal(models[0], models[1])
    # the same samples, collected in another order
    rng = np.random.default_rng(5)
    mixed = []
    for x, lab, st in reversed(train):
        k = rng.permutation(len(lab))
        mixed.append((x[k], lab[k], st[k]))
    p, _, _ = fitted(mixed, 1, path)
    same = np.mean(p == models[0])
    print(f"other order of collection: {same:.4%} of the weights equal")
    assert np.allclose(p, models[0], rtol=1e-3, atol=1e-4)
    os.unlink(path)
