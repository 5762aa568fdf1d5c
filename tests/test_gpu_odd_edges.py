"""Eigensolver steps on edges whose rows are not 16-byte aligned (n odd) or whose point count leaves
a remainder of the vector width, and with a potential that starts off a 16-byte boundary: the roots
after each step are finite and fall (a Rayleigh-Ritz step over a basis that holds the orbitals
cannot raise their sum), and the orbitals are orthonormal.

Tolerances: the sums of FP32 products carry at most 1e-6 of the largest stencil term, 204 / (24
h^2) + max|V|; the overlaps 1e-5."""
import numpy as np
import pytest
import torch

from paper_2405_01522_gb300 import rsx
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [9, 10, 13, 49])
@pytest.mark.parametrize("offset", [0, 1])
def test_steps_on_odd_edges(n, offset):
    need_gpu()
    h, k = 0.5, 3
    r = np.random.default_rng(n)
    x = (np.arange(n) - 0.5 * (n - 1)) * h
    z, y, xx = np.meshgrid(x, x, x, indexing="ij")
    flat = torch.zeros(n**3 + 4, device="cuda")
    V = flat[offset:offset + n**3].view(n, n, n)
    V.copy_(torch.tensor(0.5 * (z**2 + y**2 + xx**2) / (0.25 * n * h) ** 2))
    eig = rsx.Eigensolver(V, h, k)
    eig.init(torch.tensor(r.standard_normal((k, n, n, n))).float().cuda())
    tol = 1e-6 * (204 / (24 * h * h) + float(V.abs().max()))
    last = None
    for _ in range(4):
        theta = np.array(eig.step())
        assert np.isfinite(theta).all()
        assert last is None or theta.sum() <= last + k * tol
        last = theta.sum()
    P = eig.orbitals().double().reshape(k, -1)
    assert (P @ P.T * h**3 - torch.eye(k, device="cuda", dtype=torch.float64)).abs().max() < 1e-5
