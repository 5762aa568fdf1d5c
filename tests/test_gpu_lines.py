"""The y/z transform pass at every box edge it has a kernel for (each its own line split, CTA
shape and scratch layout), in both precisions, with the work plane in shared memory and in
global scratch: oracle parity at the library's element-wise tolerance, and the same bits
wherever the plane lives.  Three pairs make fewer work items than the grid at the small
edges; 40 pairs at 16^3 and 24^3 give every CTA several planes (the y inverse of one and the
y forward of the next share a loop)."""
import pytest
import torch

import oracle
from paper_2405_01522_gb300 import inputs, rsx
from gpu_util import TOL, need_gpu, rel_max_err, to_dev

pytestmark = pytest.mark.gpu

CASES = [(e, "fp32", 1, 3) for e in (16, 24, 32, 40, 48, 56, 64, 80, 96, 112)]
CASES += [(e, "fp64", 1, 3) for e in (16, 24, 32, 40, 48, 56, 64, 80, 96, 112)]
CASES += [(16, "fp32", 5, 8), (24, "fp32", 5, 8), (24, "fp64", 5, 8)]


@pytest.mark.parametrize("edge,prec,nocc,npsi", CASES)
def test_yz_pass_at_every_edge(edge, prec, nocc, npsi):
    need_gpu()
    shape, h = (edge, edge, 16), 0.4 if edge <= 24 else 0.3
    s = inputs.exchange_system(h=h, nocc=nocc, npsi=npsi, shape=shape, radius=1.5, seed=edge)
    ctx = rsx.Context(shape, h, prec)
    phi, psi = to_dev(s.phi, prec), to_dev(s.psi, prec)
    a = ctx.exchange_apply(phi, psi)
    ctx.set_tuning(p2_global=1)
    b = ctx.exchange_apply(phi, psi)
    ctx.sync()
    assert torch.equal(a, b)
    ref = oracle.exchange_apply(s.phi, s.psi, h)
    assert rel_max_err(a.double().cpu().numpy(), ref) < TOL[prec]
