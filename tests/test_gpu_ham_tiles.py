"""The z-marching stencil tiles through the eigensolver, against FP64: a step's residual is H psi -
theta psi of the orbitals it starts from, and the roots after one step are the Ritz values over the orbitals and their
damped-Jacobi corrections.  Edges: one tile or plane chunk and a remainder of either (4 rows, 12
planes), with and without a domain mask, an even and an odd number of sweeps.

Tolerance: a stencil value sums terms of at most A = 204 / (24 h^2) + max|V| times max|psi| through
at most 16 roundings of 2^-24; the roots see that of unit-norm orbitals, once more for the sums of
the Gram matrices."""
import numpy as np
import pytest
import torch

from paper_2405_01522_gb300 import rsx
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def laplacian4(f, h):
    out = torch.zeros_like(f)
    for ax in (1, 2, 3):
        n = f.shape[ax]
        p = torch.nn.functional.pad(f, [v for a in (3, 2, 1) for v in ((2, 2) if a == ax else (0, 0))])
        at = lambda o: p.narrow(ax, 2 + o, n)
        out += (16 * (at(1) + at(-1)) - (at(2) + at(-2)) - 30 * f) / (12 * h * h)
    return out


@pytest.mark.parametrize("n", [8, 12, 16, 28, 44])
@pytest.mark.parametrize("masked", [False, True])
@pytest.mark.parametrize("sweeps", [2, 3])
def test_residual_and_one_step_against_fp64(n, masked, sweeps):
    need_gpu()
    h, k = 0.5, 4
    r = np.random.default_rng(n)
    x = (np.arange(n) - 0.5 * (n - 1)) * h
    z, y, xx = np.meshgrid(x, x, x, indexing="ij")
    V = torch.tensor(0.5 * (z**2 + 1.3 * y**2 + 0.7 * xx**2) / (0.25 * n * h) ** 2)
    M = torch.tensor(((z**2 + y**2 + xx**2) < (0.45 * n * h) ** 2).astype(np.float64)) if masked else torch.ones(n, n, n)
    psi0 = torch.tensor(r.standard_normal((k, n, n, n)))
    eig = rsx.Eigensolver(V.float().cuda(), h, k)
    if masked:
        eig.set_mask(M.float().cuda())
    eig.init(psi0.float().cuda())
    psi = eig.orbitals().double().cpu()
    got = torch.as_tensor(eig.step(sweeps=sweeps)).double()
    res = eig.residual().double().cpu()          # of the orbitals that the step started from
    ham = lambda f, v: M * (-0.5 * laplacian4(f, h) + v * f)
    dot = lambda a, b: torch.einsum("azyx,bzyx->ab", a, b) * h**3
    Vd = V.float().double()
    tol = 16 * 2.0**-24 * (204 / (24 * h * h) + float(Vd.abs().max()))
    hp = ham(psi, Vd)
    theta = torch.diagonal(dot(psi, hp)) / torch.diagonal(dot(psi, psi))
    want = hp - theta[:, None, None, None] * psi
    assert (res - want).abs().max() < 2 * tol * psi.abs().max()

    T = (theta - torch.diagonal(dot(psi, Vd * psi))).clamp(min=0)[:, None, None, None]
    d = 3.75 / (h * h) + T
    w = want / d
    for _ in range(sweeps):
        w = w + (2.0 / 3.0) * (want - M * (-0.5 * laplacian4(w, h) + T * w)) / d
    w = w / torch.sqrt(torch.diagonal(dot(w, w)))[:, None, None, None]
    B = torch.cat([psi, w])
    S, H = dot(B, B), dot(B, ham(B, Vd))
    Li = torch.linalg.inv(torch.linalg.cholesky(S))
    ritz = torch.linalg.eigvalsh(Li @ (0.5 * (H + H.T)) @ Li.T)[:k]
    assert (got.flatten()[:k] - ritz).abs().max() < 4 * tol
