"""Device memory that a network holds for its gradients: at most what FP32 channel-first activations and
gradients take (two hidden layers forward and backward, the output and its gradient: 66 floats a
voxel) with per-block partial sums of every weight (6928 floats per 1024 voxels)."""
import pytest
import torch

from paper_2405_01522_gb300 import precond, rsx
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(12, 48, 48, 48), (64, 32, 32, 32), (32, 8, 64, 64)])
def test_gradient_workspace(shape):
    need_gpu()
    B, D, H, W = shape
    net = rsx.Net(precond.init_params(seed=5))
    tiny = torch.randn(1, 2, 8, 8, 8, device="cuda"), torch.randn(1, 8, 8, 8, device="cuda")
    net.loss_grad(*tiny, border=0)           # loads the kernels
    x, t = torch.randn(B, 2, D, H, W, device="cuda"), torch.randn(B, D, H, W, device="cuda")
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    net.loss_grad(x, t, border=0)
    used = before - torch.cuda.mem_get_info()[0]
    assert used <= (66 + 6928 / 1024) * 4 * B * D * H * W + (4 << 20)   # allocation granularity
