"""Performance cases: what a user of the library has it do, through its public
entry points, from the smallest calls to the largest.

A case is a dict of plain values; its "kind" names the work:

  step      one time step: build both hierarchies, collide (hit list), deplete
            in time order when "deplete" is set
  run       many time steps of one pair of beams as one captured run
  batch     many independent pairs of beams, many steps, as one captured run
  deplete   depletion in time order of a step's hit list
  products  electron and positron of every collision of a step's hit list
  surrogate one step of the learned statistical regime (build, cut, network)
  forward   the surrogate network on rows of node-pair features
  grad      loss and gradient of the network on a training batch
  swarm     macro-photons that can collide, split into their real photons

Beam shapes are those of the repository's workloads (Gaussian bunches in each
beam's frame, drawn here on the GPU from the seed).
"""
import ctypes
import math
import os
import struct
import tempfile

import numpy as np
import torch

from paper_1608_01125_gb300 import binding

C = 0.299792458  # um / fs
MEC2 = 0.51099895
RE = 2.8179403262e-15
KEYS = ("px", "py", "pz", "dx", "dy", "dz", "E", "w")

# transverse sigmas, longitudinal sigma [um], divergence [rad], energy spectrum,
# weights; "instance" takes its transverse sigma and median energy from the case
SHAPES = {
    "short": ((1.0, 1.0), 3.0, 5e-3, ("lognormal", 1.0, 0.5), "one"),
    "bunch": ((1.0, 1.0), 10.0, 5e-3, ("lognormal", 5.0, 0.5), "one"),
    "ellipse": ((1.0, 3.0), 15.0, 5e-3, ("gamma1.5", 20.0 / 1.5), "one"),
    "cloud": ((2.0, 2.0), 20.0, 10e-3, ("gamma2", 5.0), "uniform"),
    "instance": (None, 3.0, 5e-3, None, "one"),
    "macro": ((1.0, 1.0), 10.0, 5e-3, ("lognormal", 5.0, 0.5), "integers"),
}


def listed():
    return [
        # the smallest step: latency and launches; every pair decided in FP64
        dict(name="step_2k_fp64", kind="step", shape="short", na=2048, nb=2048, crossing=0.0,
             meet=1, dt=10.0, kappa=1e16, step=0, fp64=True, deplete=True),
        # an ordinary step: odd, unequal beams crossing at an angle, weighted photons
        dict(name="step_ragged_60deg", kind="step", shape="cloud", na=50001, nb=77773,
             crossing=1.05, meet=16, dt=20.0, kappa=1e14, step=16, fp64=False, deplete=True),
        # a large weighted head-on step of the statistical workload's shape
        dict(name="step_cloud_4m", kind="step", shape="cloud", na=4_000_000, nb=4_000_000,
             crossing=0.0, meet=16, dt=20.0, kappa=5e12, step=15, fp64=False, deplete=True),
        # the largest step: 90 degree crossing near the densest overlap
        dict(name="step_crossing90_16m", kind="step", shape="ellipse", na=1 << 24, nb=1 << 24,
             crossing=math.pi / 2, meet=128, dt=2.0, kappa=1e12, step=129, fp64=False,
             deplete=False),
        # the headline run: 2 x 1M head-on, 64 steps as one captured graph
        dict(name="run_headon_1m", kind="run", shape="bunch", na=1 << 20, nb=1 << 20,
             crossing=0.0, meet=2, dt=5.0, kappa=1e14, first=0, steps=64),
        # independent collisions of mixed sizes, angles and energies in one run
        dict(name="batch_64", kind="batch", n_inst=64, n_min=1024, n_max=131072, first=0,
             steps=16, kappa=1e14, dt=5.0),
        # depletion of the collision peak of 2 x 1M: about a million hits
        dict(name="deplete_1m", kind="deplete", shape="bunch", na=1 << 20, nb=1 << 20, dt=5.0,
             step=2, hits=1_000_000, unit=True),
        # pair products of the same hits
        dict(name="products_1m", kind="products", shape="bunch", na=1 << 20, nb=1 << 20, dt=5.0,
             step=2, hits=1_000_000),
        # one step of the learned statistical regime at 2 x 1e6
        dict(name="surrogate_1m", kind="surrogate", shape="cloud", na=1_000_000, nb=1_000_000,
             crossing=0.0, meet=16, dt=20.0, kappa=2e13, step=15, level=14),
        # inference over a step's node pairs (odd row count)
        dict(name="forward_200k", kind="forward", rows=200003),
        # one training batch of the surrogate's objective
        dict(name="grad_8k", kind="grad", rows=8192, objective=1),
        # the IP regime's split: 2 x 16384 macro-photons of 1..199 photons
        dict(name="swarm_16k", kind="swarm", shape="macro", na=16384, nb=16384, w_hi=199,
             cube=0.5, dt=5.0, kappa=1e14, first=0, steps=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "run", "batch", "deplete", "products", "surrogate",
                       "forward", "grad", "swarm"])
    if kind == "step":
        shape = rng.choice(["short", "bunch", "ellipse", "cloud"])
        na = _log(rng, 1024, 3_000_000)
        nb = max(1024, min(3_000_000, int(na * rng.uniform(0.4, 2.5))))
        dt, meet = {"short": (10.0, 1), "bunch": (5.0, 2), "ellipse": (2.0, 128),
                    "cloud": (20.0, 16)}[shape]
        kappa = {"short": 2e13, "bunch": 1e14, "ellipse": 2e14, "cloud": 2e13}[shape]
        return dict(kind=kind, shape=shape, na=na, nb=nb,
                    crossing=0.0 if rng.random() < 0.4 else rng.uniform(0.0, math.pi / 2),
                    meet=meet, dt=dt, kappa=min(1e16, kappa * 2 ** 20 / max(na, nb)),
                    step=max(0, meet + rng.randint(-2, 4)),
                    fp64=na + nb < 20000 and rng.random() < 0.4, deplete=rng.random() < 0.5)
    if kind == "run":
        n = _log(rng, 2048, 1_000_000)
        return dict(kind=kind, shape=rng.choice(["bunch", "short"]), na=n,
                    nb=max(1024, int(n * rng.uniform(0.5, 1.0))),
                    crossing=rng.choice([0.0, rng.uniform(0.0, math.pi / 2)]), meet=2, dt=5.0,
                    kappa=min(1e16, 1e14 * 2 ** 20 / n), first=rng.randint(0, 3),
                    steps=rng.randint(4, 48))
    if kind == "batch":
        return dict(kind=kind, n_inst=rng.randint(3, 60), n_min=1024,
                    n_max=_log(rng, 4096, 131072), first=rng.randint(0, 4),
                    steps=rng.randint(4, 12), kappa=1e14, dt=5.0)
    if kind in ("deplete", "products"):
        n = _log(rng, 4096, 1_000_000)
        c = dict(kind=kind, shape="bunch", na=n, nb=max(1024, int(n * rng.uniform(0.5, 1.0))),
                 dt=5.0, step=rng.randint(0, 4), hits=_log(rng, 256, n))
        if kind == "deplete":
            c["unit"] = rng.random() < 0.5
        return c
    if kind == "surrogate":
        n = _log(rng, 100_000, 1_000_000)
        return dict(kind=kind, shape="cloud", na=n, nb=n - rng.randint(0, n // 3), crossing=0.0,
                    meet=16, dt=20.0, kappa=2e13 * 1e6 / n, step=rng.randint(10, 22),
                    level=rng.choice([10, 12, 14]))
    if kind == "forward":
        return dict(kind=kind, rows=_log(rng, 1, 200_000))
    if kind == "grad":
        return dict(kind=kind, rows=_log(rng, 100, 8192), objective=rng.choice([0, 1]))
    n = _log(rng, 512, 16384)
    return dict(kind=kind, shape="macro", na=n, nb=max(256, int(n * rng.uniform(0.5, 1.0))),
                w_hi=rng.choice([3, 20, 199]), cube=rng.uniform(0.1, 1.0), dt=5.0,
                kappa=1e14, first=0, steps=rng.randint(4, 64))


# ------------------------------------------------------------------ inputs


def _gen(seed, salt):
    return torch.Generator("cuda").manual_seed(1_000_003 * int(seed) + salt)


def _energy(spec, n, g):
    f = dict(dtype=torch.float64, device="cuda", generator=g)
    if spec[0] == "lognormal":
        return torch.exp(math.log(spec[1]) + spec[2] * torch.randn(n, **f))
    e = -torch.log(1.0 - torch.rand(n, **f))
    if spec[0] == "gamma2":
        return spec[1] * (e - torch.log(1.0 - torch.rand(n, **f)))
    return spec[1] * (e + 0.5 * torch.randn(n, **f) ** 2)  # Gamma(3/2)


def _beam(n, side, g, st, sl, div, energy, weight, crossing, offset, w_hi=0):
    """A Gaussian bunch in its frame, turned into the lab: side 0 along +z, side 1
    along -z turned by `crossing` about y."""
    f = dict(dtype=torch.float64, device="cuda", generator=g)
    x, y = torch.randn(n, **f) * st[0], torch.randn(n, **f) * st[1]
    z = torch.randn(n, **f) * sl - offset
    gx, gy = torch.tan(torch.randn(n, **f) * div), torch.tan(torch.randn(n, **f) * div)
    inv = torch.rsqrt(gx * gx + gy * gy + 1.0)
    if side == 0:
        u, xp = (0.0, 0.0, 1.0), (1.0, 0.0, 0.0)
    else:
        ca, sa = math.cos(crossing), math.sin(crossing)
        u, xp = (sa, 0.0, -ca), (ca, 0.0, sa)
    yp = (0.0, 1.0, 0.0)
    out = {}
    for k, (a, b, c) in (("p", (x, y, z)), ("d", (gx * inv, gy * inv, inv))):
        for q, axis in enumerate("xyz"):
            out[k + axis] = (a * xp[q] + b * yp[q] + c * u[q]).contiguous()
    out["E"] = _energy(energy, n, g)
    if weight == "uniform":
        out["w"] = 1.0 + 9.0 * torch.rand(n, **f)
    elif weight == "integers":  # the same weights in another order
        out["w"] = (1 + torch.randperm(n, device="cuda", generator=g) % w_hi).to(torch.float64)
    else:
        out["w"] = torch.ones(n, dtype=torch.float64, device="cuda")
    return out


def _beams(case, seed):
    st, sl, div, energy, weight = SHAPES[case["shape"]]
    off = C * case.get("meet", 2) * case["dt"]
    return [_beam(case[k], q, _gen(seed, q), st, sl, div, energy, weight,
                  case.get("crossing", 0.0), off, case.get("w_hi", 0))
            for q, k in enumerate(("na", "nb"))]


def _instances(case, seed):
    """The batching workload's instances; sizes and shapes do not depend on the seed."""
    r = np.random.default_rng(17 * case["n_inst"] + case["n_max"])
    out = []
    for q in range(case["n_inst"]):
        n = int(round(math.exp(r.uniform(math.log(case["n_min"]), math.log(case["n_max"])))))
        crossing, st = r.uniform(0.0, math.pi / 2), r.uniform(0.5, 2.0)
        med = math.exp(r.uniform(math.log(0.5), math.log(50.0)))
        out.append([_beam(n, s, _gen(seed, 2 * q + s), (st, st), 3.0, 5e-3,
                          ("lognormal", med, 0.5), "one", crossing, C * 8 * case["dt"])
                    for s in (0, 1)])
    return out


def _at(b, ct):
    return [b["p" + q] + ct * b["d" + q] for q in "xyz"]


def _tstar(a, b, i, j, ct):
    pa, pb = _at(a, ct), _at(b, ct)
    dp = [pa[q][i] - pb[q][j] for q in range(3)]
    v = [C * (a["d" + q][i] - b["d" + q][j]) for q in "xyz"]
    vv = v[0] * v[0] + v[1] * v[1] + v[2] * v[2]
    return -(dp[0] * v[0] + dp[1] * v[1] + dp[2] * v[2]) / vv


def _hits(case, a, b, seed):
    """A step's hit list, as collisions leave it: case["hits"] pairs of photons that
    pass each other within the step inside one narrow transverse cell, cell by cell."""
    L = C * case["dt"]
    ct = C * case["step"] * case["dt"]
    # about twice as many pairs as wanted share a cell of this width and meet in the step
    width = math.sqrt(2.0 * case["hits"] * 250.0 / (case["na"] * case["nb"]))

    def cell(beam, shift):
        x, y, z = _at(beam, ct)
        q = [torch.floor(x / width), torch.floor(y / width),
             torch.floor((z + shift) / (2 * L))]
        q = [torch.clamp(v, -2 ** 19, 2 ** 19 - 1).to(torch.int64) + 2 ** 19 for v in q]
        return (q[0] << 40) | (q[1] << 20) | q[2]

    ca, ia = torch.sort(cell(a, L))
    cb, ib = torch.sort(cell(b, 0.0))
    lo, hi = torch.searchsorted(cb, ca), torch.searchsorted(cb, ca, right=True)
    m = hi - lo
    first = torch.cumsum(m, 0) - m
    i = torch.repeat_interleave(ia, m)
    j = ib[torch.arange(int(m.sum()), device="cuda") - torch.repeat_interleave(first - lo, m)]
    t = _tstar(a, b, i, j, ct)
    ok = torch.nonzero((t >= 0) & (t < case["dt"])).reshape(-1)
    if len(ok) < case["hits"]:
        raise RuntimeError(f"only {len(ok)} pairs meet, {case['hits']} wanted")
    pick = torch.randperm(len(ok), device="cuda", generator=_gen(seed, 20))[:case["hits"]]
    ok = ok[torch.sort(pick)[0]]
    return torch.stack([i[ok], j[ok]], 1).to(torch.int32).contiguous()


def _net(rows, seed):
    """Parameters (He initialisation, small biases), normalisation, and rows of
    features, labels and baselines as the surrogate's training meets them."""
    g = _gen(seed, 0)
    f = dict(dtype=torch.float32, device="cuda", generator=g)
    parts = []
    for k, shp in binding.MLP_ORDER:
        s = 0.1 if k.startswith("b") else math.sqrt(2.0 / shp[1])
        parts.append(torch.randn(shp, **f).reshape(-1) * s)
    norm = torch.cat([torch.randn(24, **f), 0.5 + torch.rand(24, **f)])
    x = torch.randn((rows, 24), **f) / norm[24:] + norm[:24]
    y = 6.0 * torch.rand(rows, **f) ** 2 * (torch.rand(rows, **f) < 0.7)
    return torch.cat(parts), norm, x.contiguous(), y, 4.0 * torch.rand(rows, **f)


def _model_file(level, seed):
    """A trained model as trilens_surrogate_save writes it, with drawn weights: the
    output layer small, so that the network corrects its baseline by some per cent."""
    r = np.random.default_rng(seed)
    p = [r.standard_normal(shp).reshape(-1) * (0.02 if k in ("W4", "b4") else 0.1 if k[0] == "b"
                                               else math.sqrt(2.0 / shp[1]))
         for k, shp in binding.MLP_ORDER]
    mean = np.zeros(24, np.float32)
    mean[9:13] = 3.0
    norm = np.concatenate([mean, np.full(24, 0.5, np.float32)])
    fd, path = tempfile.mkstemp(suffix=".bin")
    with os.fdopen(fd, "wb") as f:
        f.write(b"TRLSUR03" + struct.pack("<2i", level, binding.MLP_PARAMS))
        f.write(np.ones(3).tobytes() + np.ones(64).tobytes())
        f.write(norm.astype(np.float32).tobytes())
        f.write(np.concatenate(p).astype(np.float32).tobytes())
    return path


# ------------------------------------------------------------------ the passes


def prepare(case, seed):
    s = {"case": case}
    kind = case["kind"]
    if kind in ("step", "run", "surrogate"):
        a, b = _beams(case, seed)
        s["a"], s["b"] = a, b
        s["col"] = binding.Collider(a, b, case["dt"], case["kappa"],
                                    precision=binding.FP64 if case.get("fp64") else binding.FP32_BAND)
        if kind == "step":
            s["hits"] = torch.empty((8 * (case["na"] + case["nb"]) + (1 << 17), 2),
                                    dtype=torch.int32, device="cuda")
        if kind == "surrogate":
            path = _model_file(case["level"], 5)
            s["col"].surrogate_load(path)
            os.unlink(path)
    elif kind == "batch":
        s["inst"] = _instances(case, seed)
        s["col"] = binding.Batch([q[0] for q in s["inst"]], [q[1] for q in s["inst"]], case["dt"],
                                 case["kappa"])
    elif kind in ("deplete", "products"):
        a, b = _beams(case, seed)
        s["a"], s["b"], s["hits"] = a, b, _hits(case, a, b, seed)
        if kind == "deplete":
            s["col"] = binding.Collider(a, b, case["dt"], 1e14)
            s["wa"], s["wb"] = _weights(case, seed)
            s["delta"] = torch.empty(len(s["hits"]), dtype=torch.float64, device="cuda")
            s["rec"] = torch.empty(4, dtype=torch.int64, device="cuda")
        else:
            s["out"] = torch.empty((len(s["hits"]), 8), dtype=torch.float64, device="cuda")
    elif kind in ("forward", "grad"):
        s["net"] = _net(case["rows"], seed)
    else:
        s["a"], s["b"] = _beams(case, seed)
        # room for the real photons of every macro-photon, and for the offsets
        for q in "ab":
            n, m = len(s[q]["w"]), int(s[q]["w"].sum())
            s["real_" + q] = [torch.zeros(m, dtype=torch.float64, device="cuda") for _ in KEYS]
            s["owner_" + q] = torch.zeros(m, dtype=torch.int32, device="cuda")
            s["k_" + q] = torch.zeros(m, dtype=torch.int32, device="cuda")
            s["off_" + q] = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    return s


def _weights(case, seed):
    out = []
    for q, k in enumerate(("na", "nb")):
        w = torch.ones(case[k], dtype=torch.float64, device="cuda")
        if not case["unit"]:
            w = torch.exp(torch.randn(case[k], dtype=torch.float64, device="cuda",
                                      generator=_gen(seed, 10 + q)))
        out.append(w)
    return out


def _signed(v):
    return v - (1 << 64) if v >= 1 << 63 else v


def _totals(st):
    return {"count": st["count"], "weighted": np.float64(st["weighted"]),
            "hsum": _signed(st["hsum"]), "hxor": _signed(st["hxor"])}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "step":
        col, k = s["col"], case["step"]
        col.build(k)
        n = col.collide(k, s["hits"])
        out = _totals(col.stats())
        if case["deplete"]:  # the photons still left after the step
            ra, rb = s["a"]["w"].clone(), s["b"]["w"].clone()
            r = col.deplete_step(k, s["hits"], n, ra, rb)
            out.update(rem_a=ra, rem_b=rb, accepted=r["accepted"],
                       transferred=np.float64(r["transferred"]))
        return out
    if kind == "run":
        return _totals(s["col"].run(case["first"], case["steps"]))
    if kind == "batch":
        return s["col"].run(case["first"], case["steps"])
    if kind == "deplete":
        ra, rb = s["wa"].clone(), s["wb"].clone()
        s["col"].deplete_step_async(case["step"], s["hits"], len(s["hits"]), ra, rb, s["delta"],
                                    s["rec"])
        return {"rem_a": ra, "rem_b": rb, "delta": s["delta"], "accepted": s["rec"][1:2],
                "status": s["rec"][3:4], "transferred": s["rec"][0:1].view(torch.float64)}
    if kind == "products":
        return binding.pair_products(s["a"], s["b"], s["hits"], 2024, out=s["out"])
    if kind == "surrogate":
        r = s["col"].surrogate_step(case["step"], case["level"])
        return {k: np.float64(r[k]) for k in ("yield", "st_yield", "pairs", "fallback_pairs")}
    if kind == "forward":
        p, norm, x, _, _ = s["net"]
        return binding.mlp_forward(p, norm, x)
    if kind == "grad":
        p, norm, x, y, st = s["net"]
        g, loss = binding.mlp_grad(p, norm, x, y, kind=case["objective"],
                                   baseline=st if case["objective"] else None, scale=1.3)
        return {"grad": g, "loss": loss}
    # mark the macro-photons that can collide, write their photons into the caller's buffers
    lib, st = binding.lib(), ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    out = dict(zip(("mark_a", "mark_b"), binding.swarm_mark(
        s["a"], s["b"], case["cube"], case["cube"], case["dt"], case["kappa"], case["first"],
        case["steps"])))
    for q in "ab":
        mp, total = binding.beam_struct(s[q]), ctypes.c_int64(0)
        ptr = [ctypes.c_void_p(s[k + q].data_ptr()) for k in ("off_", "owner_", "k_")]
        cols = (ctypes.c_void_p * 8)(*[v.data_ptr() for v in s["real_" + q]])
        rc = lib.trilens_swarm_count(ctypes.byref(mp), ctypes.c_void_p(out["mark_" + q].data_ptr()),
                                     ptr[0], ctypes.byref(total), st)
        rc = rc or lib.trilens_swarm_expand(ctypes.byref(mp), case["cube"], ptr[0], total, cols,
                                            ptr[1], ptr[2], st)
        if rc:
            raise RuntimeError(binding.status_str(rc))
        out.update({q: s["real_" + q], "owner_" + q: s["owner_" + q], "k_" + q: s["k_" + q],
                    "total_" + q: total.value})
    return out


# ------------------------------------------------------------------ work


def work(case):
    """Each input read once and each output written once; the operations of the
    decisions or products that the results cannot do without."""
    kind = case["kind"]
    if kind in ("step", "run", "surrogate"):
        n = case["na"] + case["nb"]
        # seven FP64 values and the weight of every photon; what is left of it
        return {"bytes": n * (64 + (8 if case.get("deplete") else 0)),
                "flops": 6 * n * case.get("steps", 1)}
    if kind == "batch":
        n = 2 * case["n_inst"] * (case["n_max"] - case["n_min"]) / math.log(
            case["n_max"] / case["n_min"])
        return {"bytes": 64 * n, "flops": 6 * n * case["steps"]}
    if kind in ("deplete", "products"):
        n = case["na"] + case["nb"]
        hits = case["hits"]
        if kind == "deplete":  # positions and directions, what is left in and out, the list, delta
            return {"bytes": n * 64 + hits * 16, "flops": 35 * hits}
        return {"bytes": n * 32 + hits * 72, "flops": 81 * hits}
    macs = 24 * 128 + 2 * 128 * 128 + 128 * 2
    if kind == "forward":
        return {"bytes": case["rows"] * (24 + 2) * 4 + 4 * binding.MLP_PARAMS,
                "flops": 2 * macs * case["rows"]}
    if kind == "grad":
        return {"bytes": case["rows"] * 26 * 4 + 8 * binding.MLP_PARAMS,
                "flops": 6 * macs * case["rows"]}
    real = (case["na"] + case["nb"]) * (1 + case["w_hi"]) / 2
    return {"bytes": (case["na"] + case["nb"]) * 65 + real * (64 + 8), "flops": 6 * real}


# ------------------------------------------------------------------ the same in 64 bits


def _sigma(s):
    b = torch.sqrt(torch.clamp(s - 1.0, min=0.0) / s)
    v = (3.0 - b ** 4) * torch.log((1.0 + b) ** 2 * s) - 2.0 * b * (2.0 - b * b)
    return torch.where(s > 1.0, 0.5 * math.pi * RE * RE / s * v, torch.zeros_like(s))


def _brute(a, b, case, k):
    """Every pair of the step decided in FP64: the hits (i, j), in order of i, then j."""
    ct = C * (k * case["dt"])
    pa, pb = torch.stack(_at(a, ct)), torch.stack(_at(b, ct))
    da, db = (torch.stack([q["d" + x] for x in "xyz"]) for q in (a, b))
    out = []
    rows = max(1, (1 << 25) // pb.shape[1])
    for r in range(0, pa.shape[1], rows):
        e = slice(r, r + rows)
        v = C * (da[:, e, None] - db[:, None, :])
        p = pa[:, e, None] - pb[:, None, :]
        t = -(p * v).sum(0) / (v * v).sum(0)
        q = p + t * v
        s = a["E"][e, None] * b["E"][None, :] * (1.0 - torch.einsum("qi,qj->ij", da[:, e], db)) / (
            2.0 * MEC2 * MEC2)
        hit = (s > 1.0) & (t >= 0) & (t < case["dt"]) & (
            (q * q).sum(0) < 1e12 * case["kappa"] * _sigma(s) / math.pi)
        i, j = torch.nonzero(hit, as_tuple=True)
        out.append(torch.stack([i + r, j], 1))
    return torch.cat(out)


def _sweep(a, b, case, k, hits, ra, rb):
    """Depletion in (t*, i, j) order: what each hit takes and what is left."""
    i, j = hits[:, 0].long(), hits[:, 1].long()
    t = _tstar(a, b, i, j, C * (k * case["dt"])).cpu().numpy()
    i, j = i.cpu().numpy(), j.cpu().numpy()
    ra, rb = ra.cpu().numpy().tolist(), rb.cpu().numpy().tolist()
    delta = np.zeros(len(t))
    for h in np.lexsort((j, i, t)).tolist():
        x, y = ra[i[h]], rb[j[h]]
        d = x if x < y else y
        if d > 0.0:
            delta[h] = d
            ra[i[h]], rb[j[h]] = x - d, y - d
    return delta, np.array(ra), np.array(rb)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("step", "run"):
        steps = range(case["first"], case["first"] + case["steps"]) if kind == "run" else [case["step"]]
        if case["na"] * case["nb"] * len(steps) > 1.2e10:
            return None
        a, b = _beams(case, seed)
        out = {"count": None, "hsum": None, "hxor": None, "weighted": 0.0}
        for k in steps:
            h = _brute(a, b, case, k)
            out["weighted"] += float((a["w"][h[:, 0]] * b["w"][h[:, 1]]).sum())
        out["weighted"] = np.float64(out["weighted"])
        if case.get("deplete"):
            d, ra, rb = _sweep(a, b, case, case["step"], h, a["w"], b["w"])
            out.update(rem_a=ra, rem_b=rb, accepted=None, transferred=np.float64(d.sum()))
        return out
    if kind == "batch":
        sizes = [len(q[0]["E"]) for q in _instances(case, seed)]
        if sum(n * n for n in sizes) * case["steps"] > 1.2e10:
            return None
        return np.array([[float(sum(len(_brute(a, b, case, k)) for k in range(
            case["first"], case["first"] + case["steps"])))] * 2 for a, b in _instances(case, seed)])
    if kind == "deplete":
        a, b = _beams(case, seed)
        hits = _hits(case, a, b, seed)
        delta, ra, rb = _sweep(a, b, case, case["step"], hits, *_weights(case, seed))
        return {"rem_a": ra, "rem_b": rb, "delta": delta, "accepted": None, "status": None,
                "transferred": np.array([delta.sum()])}
    if kind == "products":
        return _exact_products(case, seed)
    if kind in ("forward", "grad"):
        return _exact_net(case, seed)
    if kind == "swarm":
        return _exact_swarm(case, seed)
    return None  # the cut is the hierarchy's own choice


def _smix(x):
    def mul(v, m):
        return v * (m - (1 << 64) if m >= 1 << 63 else m)

    def shr(v, n):
        return (v >> n) & ((1 << (64 - n)) - 1)

    z = x + (0x9E3779B97F4A7C15 - (1 << 64))
    z = mul(z ^ shr(z, 30), 0xBF58476D1CE4E5B9)
    z = mul(z ^ shr(z, 27), 0x94D049BB133111EB)
    return z ^ shr(z, 31)


def _exact_products(case, seed):
    a, b = _beams(case, seed)
    h = _hits(case, a, b, seed).long()
    i, j = h[:, 0], h[:, 1]
    e1, e2 = a["E"][i], b["E"][j]
    d1 = torch.stack([a["d" + q][i] for q in "xyz"])
    d2 = torch.stack([b["d" + q][j] for q in "xyz"])
    e, p = e1 + e2, e1 * d1 + e2 * d2
    m2 = 2.0 * e1 * e2 * (1.0 - (d1 * d2).sum(0))
    ok = m2 > 4.0 * MEC2 * MEC2
    key = 2024 ^ ((i << 32) | j)
    n = torch.zeros_like(d1)
    left = torch.ones_like(i, dtype=torch.bool)
    for t in range(0, 128, 2):
        x1, x2 = (2.0 * (((_smix(key + q) >> 11) & ((1 << 53) - 1)).double() / 2.0 ** 53) - 1.0
                  for q in (t, t + 1))
        s = x1 * x1 + x2 * x2
        take = left & (s < 1.0) & (s > 0.0)
        r = torch.sqrt(torch.clamp(1.0 - s, min=0.0))
        n = torch.where(take, torch.stack([2.0 * x1 * r, 2.0 * x2 * r, 1.0 - 2.0 * s]), n)
        left &= ~take
        if not bool(left.any()):
            break
    m2 = torch.where(ok, m2, torch.full_like(m2, 8.0 * MEC2 * MEC2))
    m = torch.sqrt(m2)
    q = torch.sqrt(0.25 * m2 - MEC2 * MEC2) * n
    beta, gamma = p / e, e / m
    out = []
    for sign in (1.0, -1.0):
        bq = (beta * (sign * q)).sum(0)
        k = gamma * gamma / (gamma + 1.0) * bq + gamma * 0.5 * m
        out.append((gamma * (0.5 * m + bq))[None])
        out.append(sign * q + beta * k)
    return torch.where(ok, torch.cat(out), torch.zeros_like(torch.cat(out))).t().contiguous()


def _exact_net(case, seed):
    p, norm, x, y, st = (v.double() for v in _net(case["rows"], seed))
    p.requires_grad_(case["kind"] == "grad")
    w, at = {}, 0
    for k, shp in binding.MLP_ORDER:
        w[k] = p[at:at + math.prod(shp)].reshape(shp)
        at += math.prod(shp)
    h = (x - norm[:24]) * norm[24:]
    for q in "123":
        z = h @ w["W" + q].t() + w["b" + q]
        h = 0.5 * z * (1.0 + torch.erf(z / math.sqrt(2.0)))
    out = h @ w["W4"].t() + w["b4"]
    if case["kind"] == "forward":
        return out
    s = torch.clamp(out[:, 1], -12.0, 12.0)
    if case["objective"]:
        base = 1.3 * st + 1.0
        mu = torch.clamp(out[:, 0], max=30.0)
        lam = base * torch.exp(mu)
        r = (torch.log1p(y) - torch.log1p(lam)).detach()
        loss = ((lam - y * torch.log(lam)) / base + 0.5 * (s + r * r * torch.exp(-s))).sum()
    else:
        loss = (0.5 * (s + (y - out[:, 0]) ** 2 * torch.exp(-s))).sum()
    (g,) = torch.autograd.grad(loss / case["rows"], p)
    return {"grad": g, "loss": loss.detach().reshape(1)}


def _exact_swarm(case, seed):
    a, b = _beams(case, seed)
    s = torch.linspace(1.5, 3.0, 300001, dtype=torch.float64, device="cuda")
    rmax = 1e6 * math.sqrt(case["kappa"] * float(_sigma(s).max()) / math.pi)
    reach = rmax + math.sqrt(0.75) * 2.0 * case["cube"]
    t0, t1 = case["first"] * case["dt"], (case["first"] + case["steps"]) * case["dt"]
    pa, pb = (torch.stack([q["p" + x] for x in "xyz"]) for q in (a, b))
    da, db = (torch.stack([q["d" + x] for x in "xyz"]) for q in (a, b))
    ma = torch.zeros(case["na"], dtype=torch.bool, device="cuda")
    mb = torch.zeros(case["nb"], dtype=torch.bool, device="cuda")
    for r in range(0, case["na"], 1024):
        e = slice(r, r + 1024)
        v = C * (da[:, e, None] - db[:, None, :])
        p = pa[:, e, None] - pb[:, None, :]
        t = torch.clamp(-(p * v).sum(0) / (v * v).sum(0), t0, t1)
        q = p + t * v
        inv = a["E"][e, None] * b["E"][None, :] * (1.0 - torch.einsum("qi,qj->ij", da[:, e], db))
        hit = ((q * q).sum(0) <= reach * reach) & (inv > 2.0 * MEC2 * MEC2)
        ma[e] |= hit.any(1)
        mb |= hit.any(0)
    g = 1.0
    for _ in range(200):
        g = (g + 1.0) ** 0.25
    out = {}
    for q, beam, m in (("a", a, ma), ("b", b, mb)):
        own = torch.nonzero(m).reshape(-1)
        w = beam["w"][own].long()
        owner = torch.repeat_interleave(own, w)
        k = torch.arange(len(owner), device="cuda") - torch.repeat_interleave(torch.cumsum(w, 0) - w, w)
        cols = []
        for d, x in enumerate(KEYS):
            v = beam[x][owner]
            if d < 3:
                u = 0.5 + k.double() * g ** -(d + 1)
                v = v + case["cube"] * (u - torch.floor(u) - 0.5)
            v = torch.ones_like(v) if x == "w" else v
            cols.append(torch.cat([v, v.new_zeros(int(beam["w"].sum()) - len(v))]))
        out[q] = cols
        out.update({"owner_" + q: None, "k_" + q: None, "mark_" + q: None, "total_" + q: None})
    return out
