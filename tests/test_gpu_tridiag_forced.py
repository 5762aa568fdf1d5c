"""The register-resident reduction by name (RSX_TRIDIAG_PATH=regs, no other path takes over): roots at the
first and last size of each tiling to FP64 accuracy (tolerances of test_gpu_tridiag.py), and a
refusal just above its range."""
import numpy as np
import pytest
import torch

import oracle
from paper_2405_01522_gb300 import rsx
from gpu_util import need_gpu

pytestmark = pytest.mark.gpu


def _solve(n):
    r = np.random.default_rng(n)
    B = r.standard_normal((n, n)) * 0.02
    eo, ev, K = np.array([-0.4]), np.linspace(-0.1, 0.5, n), B @ B.T
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    ctx = rsx.Context((16, 16, 16), 0.4, "fp64")
    w = ctx.casida_solve(d(eo), d(ev), d(K), None, 2.0, 6)
    ctx.sync()
    w_ref = np.linalg.eigvalsh(oracle.tda_matrix(eo, ev, K, None, 2.0))[:6]
    return w.cpu().numpy(), w_ref


@pytest.mark.parametrize("n", [96, 256, 257, 512, 513, 768])
def test_forced_register_path(monkeypatch, n):
    need_gpu()
    monkeypatch.setenv("RSX_TRIDIAG_PATH", "regs")
    w, w_ref = _solve(n)
    assert np.allclose(w, w_ref, rtol=0, atol=1e-12 * max(1.0, np.abs(w_ref).max()))


def test_forced_register_path_refuses_larger_matrices(monkeypatch):
    need_gpu()
    monkeypatch.setenv("RSX_TRIDIAG_PATH", "regs")
    with pytest.raises(rsx.RsxError) as err:
        _solve(769)
    assert err.value.code == rsx.RSX_EUNSUPPORTED
