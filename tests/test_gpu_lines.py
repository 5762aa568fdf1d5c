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


def _off(x, k):
    """A contiguous copy of x starting k elements into its buffer (off 16-byte boundaries)."""
    buf = torch.empty(x.numel() + k, dtype=x.dtype, device=x.device)
    buf[k:] = x.reshape(-1)
    return buf[k:].view(x.shape)


@pytest.mark.parametrize("prec,nx", [("fp32", 24), ("fp32", 40), ("fp32", 112), ("fp64", 24), ("fp64", 56)])
def test_x_passes_off_sixteen_byte_boundaries(prec, nx):
    """Orbitals and outputs that start off 16-byte boundaries take the element-wise row copies
    of the x passes: the same bits as the aligned call, for x edges of even and odd multiples of
    8 other than y's, and orbital by orbital (each pointer may be aligned or not)."""
    need_gpu()
    shape, h = (16, 16, nx), 0.4
    s = inputs.exchange_system(h=h, nocc=3, npsi=2, shape=shape, radius=1.5, seed=nx)
    ctx = rsx.Context(shape, h, prec)
    phi, psi = to_dev(s.phi, prec), to_dev(s.psi, prec)
    ref = ctx.exchange_apply(phi, psi)
    for kphi, kpsi, kout in ((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1)):
        out = _off(torch.zeros_like(psi), kout)
        got = ctx.exchange_apply(_off(phi, kphi), _off(psi, kpsi), out=out)
        ctx.sync()
        assert torch.equal(got, ref), (kphi, kpsi, kout)
    V = ctx.poisson(phi[0] * phi[0])
    rho = _off(phi[0] * phi[0], 1)
    assert torch.equal(ctx.poisson(rho, V=_off(torch.zeros_like(V), 1)), V)
    ctx.sync()


@pytest.mark.parametrize("edge,prec", [(16, "fp32"), (32, "fp32"), (32, "fp64")])
def test_back_to_back_small_solves(edge, prec):
    """Solves of at most one plane per SM are launched so that a pass's CTAs may be set up while
    the kernel before it drains.  A chain of them, each reading what a torch kernel made of the
    last result and overwriting the library's and the caller's buffers, gives the bits of the
    same chain with a synchronisation after every step; also when replayed from a CUDA graph."""
    need_gpu()
    shape, h = (edge,) * 3, 0.4
    s = inputs.exchange_system(h=h, nocc=1, npsi=1, shape=shape, radius=1.5, seed=edge)
    ctx = rsx.Context(shape, h, prec)
    phi = to_dev(s.phi, prec)

    def chain(sync):
        rho = (phi[0] * phi[0]).contiguous()
        V, seen = torch.empty_like(rho), []
        for k in range(12):
            ctx.poisson(rho, V=V)
            if sync:
                torch.cuda.synchronize()
            rho.mul_(0.5).add_(V, alpha=0.05)          # in place: the next solve's input
            ctx.exchange_apply(phi, rho.unsqueeze(0), out=V.unsqueeze(0))
            if sync:
                torch.cuda.synchronize()
            rho.sub_(V, alpha=0.1)
            seen.append(rho.clone())
        torch.cuda.synchronize()
        return seen

    ref = chain(True)
    for a, b in zip(ref, chain(False)):
        assert torch.equal(a, b)
    rho, V = (phi[0] * phi[0]).contiguous(), torch.empty_like(phi[0])
    want = ctx.poisson(rho).clone()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=side):
        ctx.poisson(rho, V=V)
        ctx.poisson(rho, V=V)
    V.zero_()
    g.replay()
    torch.cuda.synchronize()
    assert torch.equal(V, want)
