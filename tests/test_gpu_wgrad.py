"""The 3x3x3 weight and bias gradients (nn_wgrad.cuh) against the oracle where
their tiling can go wrong: rows of one and several segments, heights that are
no multiple of its row blocks, channel counts below, at and above its widths,
FP32 convolutions throughout (every parameter tensor within 1e-4 of its
largest value, as test_gpu_nn.py), and bit-identical on repeat."""
import numpy as np
import pytest

from oracle import nn as onn

from test_gpu_nn import oracle_params, rel_err

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base,levels,dims", [(1, 2, (2, 2, 2)), (2, 2, (2, 6, 64)),
                                              (3, 2, (4, 10, 62)), (5, 2, (2, 4, 126)),
                                              (7, 3, (4, 12, 20)), (14, 2, (2, 10, 8)),
                                              (15, 2, (4, 8, 8)), (16, 2, (2, 18, 4))])
def test_weight_gradients(cuda, base, levels, dims):
    import torch
    from paper_2604_18020_gb300 import mfto
    specs, params, flat = oracle_params(base, levels, seed=21)
    D, H, Wd = dims
    V = D * H * Wd
    rng = np.random.default_rng(22)
    x = rng.standard_normal((4, D, H, Wd)).astype(np.float32)
    t = rng.standard_normal((3, D, H, Wd)).astype(np.float32)
    m = (rng.random((3, D, H, Wd)) > 0.2).astype(np.float32)
    net = mfto.Net(base=base, levels=levels, max_voxels=V, max_train_voxels=V)
    net.set_params(flat)
    net.set_tensor_cores(False)
    args = [torch.tensor(a, device=cuda).reshape(-1) for a in (x, t, m)]
    loss, grad = net.gradient(*args, dims)
    loss2, grad2 = net.gradient(*args, dims)
    assert loss == loss2 and np.array_equal(grad, grad2)
    out, cache = onn.forward(params, x.astype(np.float64), levels=levels)
    loss_ref, dout = onn.mse_loss(out, t.astype(np.float64), m.astype(np.float64))
    g = onn.backward(params, cache, dout, levels=levels)
    assert abs(loss - loss_ref) <= 1e-5 * loss_ref
    at = 0
    for name, ci, co, k in specs:
        for part, size in ((name + ".w", co * ci * k ** 3), (name + ".b", co)):
            assert rel_err(grad[at:at + size], g[part].reshape(-1)) <= 1e-4, part
            at += size
