"""Lowest roots of the Tamm-Dancoff matrix at the sizes where the register-resident FP32 reduction
changes its tiling (256, 512 and 768 columns) or ends (769), one off each, and for matrices whose
reflectors vanish, against numpy's FP64 eigh of the same matrix.  The FP32 stage only supplies an
approximate eigenbasis: the FP64 corrections bring the roots to the FP64 level, so the tolerances
are those of an FP64 solve (1e-12 of the largest root's scale, residuals 1e-9)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2405_01522_gb300 import rsx
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [96, 97, 111, 255, 256, 257, 300, 511, 512, 513, 640, 767, 768, 769])
@pytest.mark.parametrize("kind", ["dense", "lowrank", "diagonal"])
def test_lowest_roots_at_tile_edges(n, kind):
    need_gpu()
    r = np.random.default_rng(n)
    B = r.standard_normal((n, n if kind == "dense" else 3)) * 0.02
    K = B @ B.T if kind != "diagonal" else np.zeros((n, n))
    eo = np.array([-0.4])
    ev = np.linspace(-0.1, 0.5, n)   # roots much farther apart than FP32 resolves
    ctx = rsx.Context((16, 16, 16), 0.4, "fp64")
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    w, X = ctx.casida_solve(d(eo), d(ev), d(K), None, 2.0, 6, vectors=True)
    ctx.sync()
    A = oracle.tda_matrix(eo, ev, K, None, 2.0)
    w_ref = np.linalg.eigvalsh(A)[:6]
    assert np.allclose(w.cpu().numpy(), w_ref, rtol=0, atol=1e-12 * max(1.0, np.abs(w_ref).max()))
    Xn = X.cpu().numpy()
    assert np.abs(A @ Xn.T - Xn.T * w_ref).max() < 1e-9
    assert np.allclose(Xn @ Xn.T, np.eye(6), atol=1e-8)
