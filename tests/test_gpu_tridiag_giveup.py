"""The register-resident reduction when its message waits run out (the spin limit 0 makes every CTA give up
at its first step, with that step's messages on their way): the kernel waits for what is in flight,
returns, and rsx_sync_status reports RSX_ETIMEOUT; with the default limit the same context then solves
the same problem to FP64 accuracy (the tolerance of test_gpu_tridiag.py)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2405_01522_gb300 import rsx
from gpu_util import need_gpu
from test_gpu_failure import _tda_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [100, 300, 640])   # 16, 32 and 48 rows a CTA
def test_message_timeout_is_reported_and_the_context_recovers(n):
    need_gpu()
    eo, ev, K = _tda_case(n)
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    ctx = rsx.Context((16, 16, 16), 0.4, "fp64")
    ctx.set_wait_limit(0)
    for _ in range(2):
        ctx.casida_solve(d(eo), d(ev), d(K), None, 1.0, 6)
        with pytest.raises(rsx.RsxError) as err:
            ctx.sync()
        assert err.value.code == rsx.RSX_ETIMEOUT
    ctx.set_wait_limit(-1)
    w = ctx.casida_solve(d(eo), d(ev), d(K), None, 1.0, 6)
    ctx.sync()
    w_ref, _ = oracle.tda_solve(oracle.tda_matrix(eo, ev, K, None, 1.0), 6)
    assert np.allclose(w.cpu().numpy(), w_ref, rtol=0, atol=1e-12)
