"""Batches of many small instances: those of at most 1024 photons share tiles of the sorted
photons, larger ones start on tiles of their own, in any order and with empty beams between.
Every instance's yield is that of the same beams in a context of their own, in a captured run
and after it step by step; the memory of tiny instances is that of their photons."""
import numpy as np
import pytest

from paper_1608_01125_gb300 import binding, synth

pytestmark = pytest.mark.gpu

DT, KAPPA, STEPS = 10.0, 1e17, 2
BIG = synth.tiny_headon(n=4096, seed=61)


@pytest.fixture(scope="module")
def pool():
    import __graft_entry__
    __graft_entry__.build()
    return tuple({k: v for k, v in binding.to_device(q).items()} for q in synth.beams(BIG))


def cut(beam, n, rng):
    at = int(rng.integers(0, BIG.a.n - n + 1))
    return {k: v[at:at + n] for k, v in beam.items()}


EDGES = [(8, 5), (1024, 1025), (1025, 1024), (0, 40), (33, 0), (31, 33), (32, 32), (2049, 3),
         (1, 2048), (64, 1024), (0, 0), (1023, 4000), (7, 7)]


@pytest.mark.parametrize("sizes", [EDGES, EDGES[::-1], "random"])
def test_yields_are_each_instance_s_own(pool, sizes):
    rng = np.random.default_rng(7)
    if sizes == "random":
        n = np.exp(rng.uniform(0, np.log(2500), (150, 2))).astype(int)
        sizes = [tuple(int(v) for v in q) for q in np.where(rng.random((150, 2)) < 0.05, 0, n)]
    A = [cut(pool[0], na, rng) for na, _ in sizes]
    B = [cut(pool[1], nb, rng) for _, nb in sizes]
    ref = np.zeros((len(sizes), 2))
    for q, (a, b) in enumerate(zip(A, B)):
        with binding.Collider(a, b, DT, KAPPA) as col:
            r = col.run(0, STEPS)
            ref[q] = r["count"], r["weighted"]
    assert (ref[:, 0] > 0).sum() > 3
    with binding.Batch(A, B, DT, KAPPA) as bt:
        assert np.array_equal(bt.run(0, STEPS), ref)
        tot = 0
        for k in range(STEPS):
            bt.build(k)
            bt.collide(k)
            tot += bt.stats()["count"]
        assert tot == ref[:, 0].sum()


def test_memory_of_tiny_instances(pool):
    import torch
    rng = np.random.default_rng(8)
    A = [cut(pool[0], 8, rng) for _ in range(8192)]
    B = [cut(pool[1], 8, rng) for _ in range(8192)]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    with binding.Batch(A, B, DT, KAPPA) as bt:
        y = bt.run(0, STEPS)
        used = free - torch.cuda.mem_get_info()[0]
    assert y.shape == (8192, 2) and y[:, 0].sum() > 0
    assert used < 200 << 20  # (a tile of 1024 photons each: 800 MB)
