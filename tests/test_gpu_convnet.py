"""The network's tensor-core kernels at the edges of their tiles: output blocks of 8 x 16 voxels
over up to 16 slices (convolutions), columns of 16 x 3 voxels over up to 32 planes (weight
gradients), boxes smaller than a halo plane, single planes and rows.  Forward, loss and
gradients against the FP64 oracle with the tolerances of test_gpu_precond.py."""
import numpy as np
import pytest
import torch

from oracle import eigensolver as oe
from paper_2405_01522_gb300 import precond, rsx
from gpu_util import need_gpu
from test_gpu_precond import unpack

pytestmark = pytest.mark.gpu

SHAPES = [(2, 1, 1, 1), (1, 2, 1, 8), (1, 16, 16, 8), (1, 17, 5, 9), (2, 33, 4, 17), (1, 18, 33, 3), (1, 3, 34, 18)]


@pytest.mark.parametrize("shape", SHAPES)
def test_network_at_tile_edges(shape):
    need_gpu()
    B, D, H, W = shape
    rng = np.random.default_rng(D * 1000 + H * 10 + W)
    p = precond.init_params(seed=5)
    net = rsx.Net(p)
    x = rng.standard_normal((B, 2, D, H, W)).astype(np.float32)
    t = rng.standard_normal((B, D, H, W)).astype(np.float32)
    out = net.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    net.sync()
    loss, g = net.loss_grad(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda(), border=0)
    params = unpack(p)
    lsum, tot = 0.0, np.zeros(len(p))
    for b in range(B):
        o, _ = oe.net_forward(x[b].astype(np.float64), params)
        assert np.max(np.abs(out[b] - o[0])) <= 2e-5 * max(1e-3, np.max(np.abs(o)))
        l_b, g_b = oe.net_loss_and_grads(x[b].astype(np.float64), t[b].astype(np.float64), params)
        lsum += l_b / B
        tot += np.concatenate([np.concatenate([gw.ravel(), gb.ravel()]) for gw, gb in g_b]) / B
    assert abs(loss - lsum) <= 1e-5 * lsum
    assert np.max(np.abs(g - tot)) <= 1e-4 * np.max(np.abs(tot))
