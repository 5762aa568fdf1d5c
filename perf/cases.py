"""The work that a user of this library has it do, as measurable cases.

The exchange action and what is built from the same pair solves come first (single-density
potential, exchange apply in both precisions, ACE, the uneven batch, Casida), then the block
eigensolver and the preconditioner network.  Sizes are those of the repository's benchmark
and tests: box edges 16 .. 112, 1 .. 24 orbitals, the 96^3 exchange step with 16 orbitals and
32 trial functions, the 80^3 Casida problem with 8 x 64 transitions, the 96^3 eigensolver with
16 bands, and the network's 32^3 training crops.
"""
import math

import numpy as np
import torch

from paper_2405_01522_gb300 import rsx

EDGES = (16, 24, 32, 40, 48, 56, 64, 80, 96, 112)
BATCH_EDGES = (48, 64, 80, 96, 112)


def listed():
    return [
        # Hartree potential of one density on a small box: the smallest call, all launch latency
        {"name": "poisson_32", "kind": "poisson", "nz": 32, "nx": 32, "prec": "fp32"},
        # the plain FP64 form that results are validated with: 4 orbitals on 32^3
        {"name": "exchange_32_fp64", "kind": "exchange", "nz": 32, "nx": 32, "prec": "fp64", "nocc": 4, "npsi": 4,
         "tuned": False},
        # a small molecule, library defaults
        {"name": "exchange_48", "kind": "exchange", "nz": 48, "nx": 48, "prec": "fp32", "nocc": 8, "npsi": 8,
         "tuned": False},
        # an elongated box whose edges are odd multiples of 8, odd orbital counts
        {"name": "exchange_40x40x56", "kind": "exchange", "nz": 40, "nx": 56, "prec": "fp32", "nocc": 5, "npsi": 7,
         "tuned": False},
        # the exchange apply of the benchmark: 512 pair solves, knobs from the autotuner
        {"name": "exchange_96", "kind": "exchange", "nz": 96, "nx": 96, "prec": "fp32", "nocc": 16, "npsi": 32,
         "tuned": True},
        # the largest box
        {"name": "exchange_112", "kind": "exchange", "nz": 112, "nx": 112, "prec": "fp32", "nocc": 6, "npsi": 8,
         "tuned": False},
        # ACE projectors of 16 orbitals and their action on 32 functions (once per SCF iteration)
        {"name": "ace_96", "kind": "ace", "nz": 96, "nx": 96, "prec": "fp32", "nocc": 16, "npsi": 32},
        # molecules of different sizes under one captured graph
        {"name": "batch_uneven", "kind": "batch", "edges": "112,96,80,80,64,64,48,48", "nocc": "6,9,14,3,20,7,24,11"},
        # excitation energies: coupling matrix of 512 transitions and its 10 lowest roots
        {"name": "casida_80", "kind": "casida", "nz": 80, "nx": 80, "nocc": 8, "nvirt": 64, "nroots": 10},
        # first iterations of the block eigensolver
        {"name": "eigensolver_96", "kind": "eig", "n": 96, "nband": 16, "steps": 2},
        # the network on the residuals of one eigensolver step
        {"name": "network_forward_96", "kind": "net_forward", "batch": 16, "d": 96, "h": 96, "w": 96},
        # one training step's loss and gradients
        {"name": "network_grad_32", "kind": "net_grad", "batch": 32, "d": 32, "h": 32, "w": 32},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(("poisson", "exchange", "exchange", "exchange", "exchange64", "ace", "batch", "casida", "eig",
                       "net_forward", "net_grad"))
    if kind == "poisson":
        return {"kind": kind, "nz": rng.choice(EDGES), "nx": rng.choice(EDGES), "prec": rng.choice(("fp32", "fp32", "fp64"))}
    if kind in ("exchange", "exchange64"):
        f64 = kind == "exchange64"
        most = 16 * 64 ** 3 if f64 else 480 * 96 ** 3       # pairs x points
        nz, nx = rng.choice(EDGES[:7] if f64 else EDGES), rng.choice(EDGES[:7] if f64 else EDGES)
        pairs = max(1, min(640, most // (nz * nz * nx)))
        nocc = _log_int(rng, 1, min(16, pairs))
        return {"kind": "exchange", "nz": nz, "nx": nx, "prec": "fp64" if f64 else "fp32", "nocc": nocc,
                "npsi": _log_int(rng, 1, max(1, min(40, pairs // nocc))), "tuned": (not f64) and rng.random() < 0.25}
    if kind == "ace":
        nz, nx = rng.choice(EDGES[2:]), rng.choice(EDGES[2:])
        return {"kind": kind, "nz": nz, "nx": nx, "prec": "fp32", "nocc": _log_int(rng, 2, 20), "npsi": _log_int(rng, 1, 40)}
    if kind == "batch":
        m = rng.randint(2, 4)
        return {"kind": kind, "edges": ",".join(str(rng.choice(BATCH_EDGES)) for _ in range(m)),
                "nocc": ",".join(str(rng.randint(2, 12)) for _ in range(m))}
    if kind == "casida":
        nocc, nvirt = rng.randint(2, 8), _log_int(rng, 6, 60)
        return {"kind": kind, "nz": rng.choice(EDGES[2:7]), "nx": rng.choice(EDGES[2:7]), "nocc": nocc, "nvirt": nvirt,
                "nroots": min(10, nocc * nvirt)}
    if kind == "eig":
        return {"kind": kind, "n": rng.choice((24, 30, 40, 49, 64, 80, 96)), "nband": rng.randint(2, 16), "steps": rng.randint(1, 2)}
    b = _log_int(rng, 1, 12)
    lo, hi = (8, 33) if kind == "net_grad" else (9, 80)
    return {"kind": kind, "batch": b, "d": rng.randint(lo, hi), "h": rng.randint(lo, hi), "w": rng.randint(lo, hi)}


# ------------------------------------------------------------------------------- inputs
def _spacing(n):
    return 0.2 if n >= 80 else 0.3 if n >= 32 else 0.4


def _rand(gen, *shape, lo=0.0, hi=1.0):
    return lo + (hi - lo) * torch.rand(*shape, generator=gen, dtype=torch.float64)


def _ball(gen, n, radius):
    """n points in a ball: uniform directions, cube-root radii."""
    v = torch.randn(n, 3, generator=gen, dtype=torch.float64)
    return radius * _rand(gen, n, 1) ** (1 / 3) * v / v.norm(dim=1, keepdim=True)


def _gaussian_sums(gen, norb, shape, h, alpha, radius, nterm=3):
    """Orbitals as sums of s-type Gaussians, own centres, exponents and coefficients (FP64, on the GPU)."""
    cen = _ball(gen, norb * nterm, radius).cuda()
    a = _rand(gen, norb * nterm, lo=alpha[0], hi=alpha[1]).cuda()
    c = _rand(gen, norb * nterm, lo=0.3, hi=1.0).cuda() * (torch.randint(0, 2, (norb * nterm,), generator=gen) * 2 - 1).cuda()
    f = []
    for ax, n in zip((2, 1, 0), shape):
        r = (torch.arange(n, dtype=torch.float64, device="cuda") - n / 2) * h
        f.append(torch.exp(-a[:, None] * (r[None, :] - cen[:, ax:ax + 1]) ** 2).view(norb, nterm, n))
    f[0] = f[0] * c.view(norb, nterm, 1)
    out = torch.empty((norb,) + tuple(shape), dtype=torch.float64, device="cuda")
    for k in range(norb):
        yx = f[1][k][:, :, None] * f[2][k][:, None, :]
        out[k] = torch.einsum("gz,gyx->zyx", f[0][k], yx)
    return out


def _orthonormal(f, h):
    v = f.reshape(f.shape[0], -1)
    for _ in range(2):
        s = h ** 3 * (v @ v.T)
        v = torch.linalg.inv(torch.linalg.cholesky(s)) @ v
    return v.reshape(f.shape)


def _normalised(f, h):
    v = f.reshape(f.shape[0], -1)
    return (v / (h ** 1.5 * v.norm(dim=1, keepdim=True))).reshape(f.shape)


def _orbital_inputs(case, seed):
    """(shape, h, phi orthonormal, psi normalised) in the case's precision."""
    gen = torch.Generator().manual_seed(seed)
    shape = (case["nz"], case["nz"], case["nx"])
    h = _spacing(case["nz"])
    radius = 0.18 * h * min(shape)
    alpha = (0.3, 3.0) if h <= 0.3 else (0.5, 2.0)
    dt = torch.float32 if case.get("prec", "fp32") == "fp32" else torch.float64
    phi = _orthonormal(_gaussian_sums(gen, case["nocc"], shape, h, alpha, radius), h).to(dt)
    psi = None
    if case.get("npsi"):
        psi = _normalised(_gaussian_sums(gen, case["npsi"], shape, h, alpha, radius), h).to(dt)
    return shape, h, phi, psi


def _density(case, seed):
    gen = torch.Generator().manual_seed(seed)
    shape = (case["nz"], case["nz"], case["nx"])
    h = _spacing(case["nz"])
    f = _normalised(_gaussian_sums(gen, 2, shape, h, (0.3, 2.0), 0.18 * h * min(shape)), h)
    rho = 2.0 * (f * f).sum(dim=0)
    return shape, h, rho.to(torch.float32 if case["prec"] == "fp32" else torch.float64).contiguous()


def _molecules(case, seed):
    out = []
    for m, (e, k) in enumerate(zip(case["edges"].split(","), case["nocc"].split(","))):
        gen = torch.Generator().manual_seed(seed * 1009 + m)
        e, k, h = int(e), int(k), 0.2
        phi = _orthonormal(_gaussian_sums(gen, k, (e, e, e), h, (0.3, 3.0), 0.16 * h * e), h)
        out.append(phi.float())
    return out


def _casida_inputs(case, seed):
    gen = torch.Generator().manual_seed(seed)
    shape = (case["nz"], case["nz"], case["nx"])
    h = 0.25 if case["nz"] >= 80 else _spacing(case["nz"])
    no, nv = case["nocc"], case["nvirt"]
    allorb = _orthonormal(_gaussian_sums(gen, no + nv, shape, h, (0.3, 3.0), 0.18 * h * min(shape)), h).float()
    eo = torch.sort(_rand(gen, no, lo=-0.8, hi=-0.3)).values.cuda()
    ev = torch.sort(_rand(gen, nv, lo=-0.1, hi=0.5)).values.cuda()
    return shape, h, allorb[:no].contiguous(), allorb[no:].contiguous(), eo, ev


def _eig_inputs(case, seed):
    """Smooth model atoms (error-function wells) and Gaussian-sum starting orbitals."""
    gen = torch.Generator().manual_seed(seed)
    n, h = case["n"], 0.2 if case["n"] >= 64 else 0.4
    radius = 0.15 * n * h
    r = (torch.arange(n, dtype=torch.float64, device="cuda") - n / 2) * h
    V = torch.zeros(n, n, n, dtype=torch.float64, device="cuda")
    for X, Y, Z in _ball(gen, 4, radius).tolist():
        d = torch.sqrt((r[:, None, None] - Z) ** 2 + (r[None, :, None] - Y) ** 2 + (r[None, None, :] - X) ** 2)
        V -= 4.0 * torch.erf(d / 0.6) / d.clamp_min(1e-9)
    psi = _normalised(_gaussian_sums(gen, case["nband"], (n, n, n), h, (0.3, 1.5), radius), h)
    return h, V.float(), psi.float()


_NET_SHAPES = ((16, 2, 27), (16,), (16, 16, 27), (16,), (1, 16, 27), (1,))


def _net_inputs(case, seed):
    """He-initialised parameters, normalised residual-like channel and a potential channel."""
    gen = torch.Generator().manual_seed(seed)
    parts = []
    for s in _NET_SHAPES:
        if len(s) == 3:
            parts.append(torch.randn(*s, generator=gen, dtype=torch.float64) * math.sqrt(2.0 / (s[1] * s[2])))
        else:
            parts.append(0.05 * torch.randn(*s, generator=gen, dtype=torch.float64))
    p = torch.cat([t.reshape(-1) for t in parts]).float()
    g = torch.Generator(device="cuda").manual_seed(seed)
    size = (case["batch"], 2, case["d"], case["h"], case["w"])
    x = torch.randn(*size, generator=g, device="cuda")
    x[:, 1] = -torch.rand(size[:1] + size[2:], generator=g, device="cuda")
    target = 0.1 * torch.randn(size[:1] + size[2:], generator=g, device="cuda")
    return p, x, target


# ---------------------------------------------------------------------------- the calls
def prepare(case, seed):
    kind = case["kind"]
    if kind == "poisson":
        shape, h, rho = _density(case, seed)
        return {"kind": kind, "ctx": rsx.Context(shape, h, case["prec"]), "rho": rho}
    if kind in ("exchange", "ace"):
        shape, h, phi, psi = _orbital_inputs(case, seed)
        ctx = rsx.Context(shape, h, case["prec"])
        if case.get("tuned"):
            ctx.autotune(case["nocc"], case["npsi"])
        return {"kind": kind, "ctx": ctx, "phi": phi, "psi": psi}
    if kind == "batch":
        phi = _molecules(case, seed)
        W, xi = [torch.empty_like(p) for p in phi], [torch.empty_like(p) for p in phi]
        b = rsx.Batch([p.shape[1] for p in phi], [p.shape[0] for p in phi], 0.2)
        b.bind(phi, W, xi)
        return {"kind": kind, "batch": b, "W": W, "xi": xi}
    if kind == "casida":
        shape, h, occ, virt, eo, ev = _casida_inputs(case, seed)
        return {"kind": kind, "ctx": rsx.Context(shape, h, "fp32"), "occ": occ, "virt": virt, "eo": eo, "ev": ev,
                "nroots": case["nroots"]}
    if kind == "eig":
        h, V, psi = _eig_inputs(case, seed)
        return {"kind": kind, "eig": rsx.Eigensolver(V, h, case["nband"]), "psi": psi, "steps": case["steps"]}
    p, x, target = _net_inputs(case, seed)
    return {"kind": kind, "net": rsx.Net(p.numpy()), "x": x, "target": target}


def run(state):
    kind = state["kind"]
    if kind == "poisson":
        return state["ctx"].poisson(state["rho"])
    if kind == "exchange":
        return state["ctx"].exchange_apply(state["phi"], state["psi"])
    if kind == "ace":
        xi = state["ctx"].ace_build(state["phi"])
        return {"xi": xi, "vpsi": state["ctx"].ace_apply(xi, state["psi"])}
    if kind == "batch":
        state["batch"].run()
        return {"W": state["W"], "xi": state["xi"]}
    if kind == "casida":
        K = state["ctx"].casida_K(state["occ"], state["virt"])
        omega = state["ctx"].casida_solve(state["eo"], state["ev"], K, delta_M=2.0, nroots=state["nroots"])
        return {"omega": omega.tolist()}          # the excitation energies, read on the host
    if kind == "eig":
        eig = state["eig"]
        eig.init(state["psi"])
        for _ in range(state["steps"]):
            theta = eig.step()
        return {"theta": theta, "orbitals": eig.orbitals(), "residual": eig.residual()}
    if kind == "net_forward":
        return state["net"].forward(state["x"])
    loss, grad = state["net"].loss_grad(state["x"], state["target"], border=3 if min(state["x"].shape[2:]) > 8 else 1)
    return {"loss": loss, "grad": grad}


# --------------------------------------------------------------------- least work of a call
def _solve_flops(nz, ny, nx):
    """One pair solve by a zero-padded FFT convolution, forward and back, with the transforms of
    all-zero lines and of discarded lines left out (5 M log2 M real operations per complex line)."""
    line = lambda m: 5.0 * m * math.log2(m)
    hx = nx + 1
    return 2.0 * (nz * ny / 2 * line(2 * nx) + hx * nz * line(2 * ny) + hx * 2 * ny * line(2 * nz)) + 2.0 * nx * ny * nz


def work(case):
    kind = case["kind"]
    es = 8 if case.get("prec") == "fp64" else 4
    if kind == "poisson":
        n = case["nz"] ** 2 * case["nx"]
        return {"bytes": 2 * n * es, "flops": _solve_flops(case["nz"], case["nz"], case["nx"])}
    if kind == "exchange":
        n = case["nz"] ** 2 * case["nx"]
        pairs = case["nocc"] * case["npsi"]
        return {"bytes": (case["nocc"] + 2 * case["npsi"]) * n * es,
                "flops": pairs * (_solve_flops(case["nz"], case["nz"], case["nx"]) + 3 * n)}
    if kind == "ace":
        n, k, p = case["nz"] ** 2 * case["nx"], case["nocc"], case["npsi"]
        return {"bytes": (2 * k + 2 * p) * n * es,
                "flops": k * (k + 1) / 2 * _solve_flops(case["nz"], case["nz"], case["nx"]) + 2.0 * n * (4 * k * k / 2 + 2 * k * p)}
    if kind == "batch":
        b = f = 0.0
        for e, k in zip(case["edges"].split(","), case["nocc"].split(",")):
            e, k = int(e), int(k)
            b += 3 * k * e ** 3 * 4
            f += k * (k + 1) / 2 * _solve_flops(e, e, e) + 4.0 * k * k * e ** 3
        return {"bytes": b, "flops": f}
    if kind == "casida":
        nz, nx, nt = case["nz"], case["nx"], case["nocc"] * case["nvirt"]
        return {"bytes": (case["nocc"] + case["nvirt"]) * nz * nz * nx * 4 + 8 * nt * nt,
                "flops": nt * _solve_flops(nz, nz, nx) / 2 + 1.0 * nt * nt * nz * nz * nx + 4.0 / 3.0 * nt ** 3}
    if kind == "eig":
        n, k = case["n"] ** 3, case["nband"]
        # a step reads and writes the orbitals, the preconditioned residuals and the directions once
        return {"bytes": 4.0 * n * (2 * k + 1 + case["steps"] * 6 * k), "flops": case["steps"] * n * (2.0 * 2 * (3 * k) ** 2 + 6 * 25 * k)}
    v = case["batch"] * case["d"] * case["h"] * case["w"]
    mac = 27 * (2 * 16 + 16 * 16 + 16)
    return {"bytes": 4.0 * v * 3, "flops": 2.0 * v * mac * (1 if kind == "net_forward" else 3)}


# -------------------------------------------------------------------------- 64-bit values
def _kernel_hat(shape, h):
    """DFT of 1 / |r| (cell average at 0) on the doubled box, real half spectrum along x."""
    ax = [torch.minimum(torch.arange(2 * n, device="cuda"), 2 * n - torch.arange(2 * n, device="cuda")).double() for n in shape]
    r = torch.sqrt(ax[0][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[2][None, None, :] ** 2)
    g = 1.0 / (h * r)
    g[0, 0, 0] = (3.0 * math.log(2.0 + math.sqrt(3.0)) - 0.5 * math.pi) / h
    return torch.fft.rfftn(g).real.contiguous()


def _potential(rho, ghat, h):
    nz, ny, nx = rho.shape
    f = torch.fft.rfftn(rho, s=(2 * nz, 2 * ny, 2 * nx)) * ghat
    return h ** 3 * torch.fft.irfftn(f, s=(2 * nz, 2 * ny, 2 * nx))[:nz, :ny, :nx]


def _exact_exchange(phi, psi, h, sym=False):
    phi, psi = phi.double(), psi.double()
    ghat = _kernel_hat(phi.shape[1:], h)
    out = torch.zeros_like(psi)
    for p in range(psi.shape[0]):
        for j in range(p if sym else 0, phi.shape[0]):
            v = _potential(phi[j] * psi[p], ghat, h)
            out[p] -= phi[j] * v
            if sym and j != p:
                out[j] -= phi[p] * v
    return out


def _exact_xi(phi, w, h):
    p, v = phi.double().reshape(phi.shape[0], -1), w.reshape(w.shape[0], -1)
    m = h ** 3 * (p @ v.T)
    low = torch.linalg.cholesky(-0.5 * (m + m.T))
    return (torch.linalg.inv(low) @ v).reshape(w.shape)


def _conv(x, w, b):
    """3^3 convolution with zero padding, tap by tap; x [B][C][D][H][W], w [O][C][27]."""
    xp = torch.nn.functional.pad(x, (1, 1, 1, 1, 1, 1))
    d, hh, ww = x.shape[2:]
    out = b.view(1, -1, 1, 1, 1).expand(x.shape[0], -1, d, hh, ww)
    for t in range(27):
        z, y, c = t // 9, t // 3 % 3, t % 3
        out = out + torch.einsum("oc,bcdhw->bodhw", w[:, :, t], xp[:, :, z:z + d, y:y + hh, c:c + ww])
    return out


def _net_params(p):
    out, o = [], 0
    for s in _NET_SHAPES:
        n = math.prod(s)
        t = p[o:o + n].view(s)
        o += n
        out.append((t.bfloat16() if len(s) == 3 else t).double().cuda())   # weights are used in bf16
    return out


def _net(x, q):
    a = torch.relu(_conv(x, q[0], q[1]))
    a = torch.relu(_conv(a, q[2], q[3]))
    return _conv(a, q[4], q[5])[:, 0]


def _laplacian(f, h):
    out = torch.zeros_like(f)
    for ax in (1, 2, 3):
        g = torch.nn.functional.pad(f.transpose(ax, 3), (2, 2))
        n = g.shape[3] - 4
        out += ((-g[..., :n] + 16 * g[..., 1:n + 1] - 30 * g[..., 2:n + 2] + 16 * g[..., 3:n + 3] - g[..., 4:]) / (12 * h * h)).transpose(ax, 3)
    return out


def _exact_theta(case, seed):
    """Ritz values of the same block iteration in 64 bits: [Psi | W], then [Psi | W | P]."""
    h, V, psi = _eig_inputs(case, seed)
    V, psi = V.double(), psi.double()
    k, shape = psi.shape[0], psi.shape
    ham = lambda f: -0.5 * _laplacian(f, h) + V * f

    def ritz(basis):
        b, hb = basis.reshape(basis.shape[0], -1), ham(basis).reshape(basis.shape[0], -1)
        s, hs = (h ** 3 * (b @ b.T)).cpu(), (h ** 3 * (b @ hb.T)).cpu()
        li = torch.linalg.inv(torch.linalg.cholesky(0.5 * (s + s.T)))
        t, y = torch.linalg.eigh(li @ (0.5 * (hs + hs.T)) @ li.T)
        q = (li.T @ y[:, :k]).T.contiguous()
        tail = (q[:, k:].cuda() @ b[k:]).reshape(shape) if basis.shape[0] > k else None
        return t[:k], (q.cuda() @ b).reshape(shape), tail

    theta, psi, tail = ritz(psi)
    for _ in range(case["steps"]):
        t = theta.cuda().view(-1, 1, 1, 1)
        res = ham(psi) - t * psi
        kin = t - (h ** 3 * (psi * psi * V).sum(dim=(1, 2, 3))).view(-1, 1, 1, 1)
        d = 3.75 / h ** 2 + kin
        w = res / d
        for _ in range(3):
            w = w + (2.0 / 3.0) * (res + 0.5 * _laplacian(w, h) - kin * w) / d
        rows = [psi, _normalised(w, h)] + ([_normalised(tail, h)] if tail is not None else [])
        theta, psi, tail = ritz(torch.cat(rows))
    return theta.tolist()


def exact(case, seed):
    kind = case["kind"]
    if kind == "poisson":
        shape, h, rho = _density(case, seed)
        return _potential(rho.double(), _kernel_hat(shape, h), h)
    if kind == "exchange":
        _, h, phi, psi = _orbital_inputs(case, seed)
        return _exact_exchange(phi, psi, h)
    if kind == "ace":
        _, h, phi, psi = _orbital_inputs(case, seed)
        xi = _exact_xi(phi, _exact_exchange(phi, phi, h, sym=True), h)
        x, p = xi.reshape(xi.shape[0], -1), psi.double().reshape(psi.shape[0], -1)
        return {"xi": xi, "vpsi": -((h ** 3 * (p @ x.T)) @ x).reshape(psi.shape)}
    if kind == "batch":
        phi = _molecules(case, seed)
        W = [_exact_exchange(p, p, 0.2, sym=True) for p in phi]
        return {"W": W, "xi": [_exact_xi(p, w, 0.2) for p, w in zip(phi, W)]}
    if kind == "casida":
        shape, h, occ, virt, eo, ev = _casida_inputs(case, seed)
        ghat = _kernel_hat(shape, h)
        rho = (occ.double()[:, None] * virt.double()[None, :]).reshape((-1,) + tuple(shape))
        v = torch.empty_like(rho)
        for t in range(rho.shape[0]):
            v[t] = _potential(rho[t], ghat, h)
        K = h ** 3 * (rho.reshape(rho.shape[0], -1) @ v.reshape(v.shape[0], -1).T)
        A = torch.diag((ev[None, :] - eo[:, None]).reshape(-1)) + 2.0 * 0.5 * (K + K.T)
        return {"omega": np.linalg.eigvalsh(A.cpu().numpy())[:case["nroots"]].tolist()}
    if kind == "eig":
        return {"theta": _exact_theta(case, seed), "orbitals": None, "residual": None}
    p, x, target = _net_inputs(case, seed)
    q = _net_params(p)
    if kind == "net_forward":
        return torch.cat([_net(x[b:b + 1].double(), q) for b in range(x.shape[0])])
    for t in q:
        t.requires_grad_(True)
    c = 3 if min(x.shape[2:]) > 8 else 1
    count = x.shape[0] * math.prod(n - 2 * c for n in x.shape[2:])
    loss = 0.0
    for b in range(x.shape[0]):
        diff = (_net(x[b:b + 1].double(), q) - target[b:b + 1].double())[:, c:-c, c:-c, c:-c]
        part = diff.square().sum() / count
        part.backward()
        loss += part.item()
    return {"loss": loss, "grad": torch.cat([t.grad.reshape(-1) for t in q]).cpu().numpy()}
