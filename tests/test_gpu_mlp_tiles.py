"""The network's kernels where their loops turn over: more tiles of 128 rows than
blocks (gradients) and than groups of all blocks (inference), and calls from several
threads and streams at once.  Tolerances as in test_gpu_mlp.py."""
import threading

import numpy as np
import pytest

from oracle import mlp
from paper_1608_01125_gb300 import binding
from test_gpu_mlp import _check_grads, _setup

pytestmark = pytest.mark.gpu


def _sms():
    import torch
    return torch.cuda.get_device_properties(0).multi_processor_count


def test_gradients_with_more_tiles_than_blocks():
    m = 128 * _sms() + 129  # block 0 and 1 take a second tile, the last one ragged
    p, x, y, P, N, X, Y = _setup(m, 11)
    g, loss = binding.mlp_grad(P, N, X, Y)
    L, gref = mlp.loss_and_grads(p, x, y)
    assert abs(float(loss.item()) / m - L) <= 0.03 * abs(L) + 1e-3
    _check_grads(binding.mlp_unflatten(g.cpu().numpy().astype(np.float64)), gref)


def test_forward_with_more_tiles_than_groups():
    m = 4 * 128 * _sms() + 130
    p, x, y, P, N, X, Y = _setup(m, 12)
    out = binding.mlp_forward(P, N, X).cpu().numpy()
    ref, _ = mlp.forward(p, x)
    err = np.abs(out - ref)
    scale = np.abs(ref).mean() + 1e-3
    assert err.max() <= 0.08 * scale + 0.05 * np.abs(ref).max()
    # a row's output does not depend on the tile it falls into
    tail = binding.mlp_forward(P, N, X[-300:].contiguous()).cpu().numpy()
    assert np.array_equal(out[-300:], tail)


def test_calls_from_several_threads_and_streams():
    import torch
    m = 3000
    p, x, y, P, N, X, Y = _setup(m, 13)
    ref_o = binding.mlp_forward(P, N, X).cpu().numpy()
    ref_g = binding.mlp_grad(P, N, X, Y)[0].cpu().numpy()
    bad = []

    def work():
        st = torch.cuda.Stream()
        with torch.cuda.stream(st):
            for _ in range(20):
                o = binding.mlp_forward(P, N, X, stream=st)
                g, _ = binding.mlp_grad(P, N, X, Y, stream=st)
                st.synchronize()
                if not (np.array_equal(o.cpu().numpy(), ref_o)
                        and np.array_equal(g.cpu().numpy(), ref_g)):
                    bad.append(1)

    ts = [threading.Thread(target=work) for _ in range(4)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad
