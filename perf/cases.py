"""Measured cases: the work a user of the library has it do, through the public binding.

Kinds of a case (``kind``):

* ``apply``     the matrix-free operator on a batch of fields (helm_apply, H or the shifted Laplacian);
* ``residual``  the FP64 residual of a batch of complex128 iterates (helm_residual), every restart's check;
* ``vcycle``    one multigrid V-cycle (helm_vcycle), the preconditioner of every FGMRES step;
* ``samples``   training pairs of a medium: FGMRES with a fixed number of steps per right-hand side
                (cnn_make_samples), i.e. Arnoldi, V-cycles, update and residual without a stopping test;
* ``solve``     helm_solve to a tolerance, forward or adjoint, several frequencies in one batch;
* ``misfit``    the FWI misfit and its gradient (fwi_misfit_grad): forward and adjoint solves;
* ``precond``   the encoder-solver network preconditioner with its V-cycle (cnn_precond_apply);
* ``loss_grad`` the training loss and the gradient of every network parameter (cnn_loss_grad).

Media are layered with smoothed noise, 1.5-4.5 km/s, with a quadratic absorbing layer on three sides;
grids have about ten points per 1.5 km/s wavelength at the largest frequency.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch
import torch.nn.functional as F

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TRAINED = os.path.join(ROOT, "paper_2405_17696_gb300", "weights", "encoder_solver_1024x512_8hz.ckpt")
CKPT_HEADER_BYTES = 80     # include/helm.h, cnn_save
WIDTHS = (16, 32, 64, 128)


def _case(kind, nx, nz, hx, hz, freqs, nrhs, **more):
    return {"kind": kind, "nx": nx, "nz": nz, "hx": hx, "hz": hz, "freqs": freqs, "nrhs": nrhs, **more}


def listed():
    return [
        # the preconditioner for one source on the smallest configuration: launches and latency
        dict(name="vcycle_160x160_1rhs", **_case("vcycle", 160, 160, 25.0, 25.0, "6", 1)),
        # one operator application on the batched configuration
        dict(name="apply_512x256_192rhs", **_case("apply", 512, 256, 20.0, 20.0, "3,4.5,6", 192, op=0)),
        # the restart check of the batched configuration
        dict(name="residual_512x256_192rhs", **_case("residual", 512, 256, 20.0, 20.0, "3,4.5,6", 192)),
        # the preconditioner of every FGMRES step of the batched configuration
        dict(name="vcycle_512x256_192rhs", **_case("vcycle", 512, 256, 20.0, 20.0, "3,4.5,6", 192)),
        # the largest window grid of the full-FWI configuration (10 Hz): ragged tiles, hx != hz
        dict(name="vcycle_1360x688_40rhs",
             **_case("vcycle", 1360, 688, 2048 * 10.0 / 1360, 1024 * 10.0 / 688, "10", 40)),
        # Eq. 4.3 training pairs on the network's medium size
        dict(name="samples_1024x512_16rhs", **_case("samples", 1024, 512, 12.5, 12.5, "8", 16)),
        # one source of the smallest configuration solved: what a single small solve waits for
        dict(name="solve_160x160_1rhs", **_case("solve", 160, 160, 25.0, 25.0, "6", 1, tol=1e-8, adjoint=False)),
        # the batched configuration: 64 sources at three frequencies
        dict(name="solve_512x256_192rhs",
             **_case("solve", 512, 256, 20.0, 20.0, "3,4.5,6", 192, tol=1e-8, adjoint=False)),
        # the lowest window of the full-FWI configuration: misfit and gradient, small anisotropic grid
        dict(name="misfit_336x176_32src",
             **_case("misfit", 336, 176, 2048 * 10.0 / 336, 1024 * 10.0 / 176, "2.5", 32, nrcv=84, tol=1e-8)),
        # the network preconditioner on a small grid: 29 convolution layers, launches and latency
        dict(name="precond_128x64_16rhs", **_case("precond", 128, 64, 20.0, 20.0, "6", 16, weights="trained")),
        # the network preconditioner on the configuration the network is specified on
        dict(name="precond_1024x512_32rhs", **_case("precond", 1024, 512, 12.5, 12.5, "8", 32, weights="trained")),
        # one training step's loss and gradient on that configuration, batch 16
        dict(name="loss_grad_1024x512_16rhs",
             **_case("loss_grad", 1024, 512, 12.5, 12.5, "8", 16, weights="seeded")),
    ]


def draw(rng):
    kind = rng.choice(["apply", "residual", "vcycle", "vcycle", "samples", "solve", "misfit", "precond", "loss_grad"])

    def log(lo, hi):
        return math.exp(rng.uniform(math.log(lo), math.log(hi)))

    # per kind: range of nx, multiple that nz is of, largest right-hand-side count, largest nx nz nrhs
    lo, hi, div, most, points = {
        "apply": (64, 1360, 4, 256, 25e6), "residual": (64, 1360, 4, 256, 25e6), "vcycle": (64, 1360, 4, 256, 25e6),
        "samples": (64, 1024, 4, 64, 8e6), "solve": (64, 400, 4, 96, 3e6), "misfit": (64, 336, 4, 64, 2e6),
        "precond": (64, 1024, 8, 64, 16e6), "loss_grad": (64, 1024, 8, 32, 8e6)}[kind]
    nx = max(lo, int(log(lo, hi)) // 8 * 8)
    nz = max(32, int(nx * rng.uniform(0.4, 1.0)) // div * div)
    nrhs = max(1, int(log(1, most + 1)))
    nrhs = max(1, min(nrhs, most, int(points / (nx * nz))))
    fmax = rng.uniform(2.5, 10.0)
    hx = 150.0 / fmax
    hz = hx * rng.choice([1.0, 1.0, rng.uniform(0.9, 1.1)])
    nfreq = rng.choice([1, 1, 2, 3])
    freqs = ",".join("%.3g" % (fmax * (1.0 - 0.5 * j / nfreq)) for j in reversed(range(nfreq)))
    c = _case(kind, nx, nz, hx, hz, freqs, nrhs)
    if kind == "apply":
        c["op"] = rng.choice([0, 1])
    if kind in ("solve", "misfit"):
        c["tol"] = 1e-8
    if kind == "solve":
        c["adjoint"] = rng.choice([False, True])
    if kind == "misfit":
        c["nrcv"] = rng.randrange(8, nx // 4 + 1)
    if kind in ("precond", "loss_grad"):
        c["weights"] = "trained" if kind == "precond" else "seeded"   # a solve's network, and a training's start
    return c


# ---- inputs ---------------------------------------------------------------------------

def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _freqs(case):
    return [float(f) for f in case["freqs"].split(",")]


def _nsys(case):
    """Right-hand sides of one solver batch (a misfit's sources at every frequency)."""
    return case["nrhs"] * (len(_freqs(case)) if case["kind"] == "misfit" else 1)


def _cn(g, shape, dev, dtype=torch.complex64):
    return torch.randn(shape, generator=g, device=dev, dtype=dtype)


def _medium(case, g, dev):
    """kappa = 1/c of a layered medium with smoothed noise, and the absorbing layer (float32 [nz][nx])."""
    nx, nz = case["nx"], case["nz"]
    x = torch.arange(nx, device=dev, dtype=torch.float64)
    z = torch.arange(nz, device=dev, dtype=torch.float64)[:, None]
    u = torch.rand((12, 3), generator=g, device=dev, dtype=torch.float64)
    top = (torch.arange(12, device=dev)[:, None] * (nz / 12.0)
           + u[:, :1] * (nz / 48.0) * torch.sin(2 * math.pi * (x / ((0.25 + 0.75 * u[:, 1:2]) * nx) + u[:, 2:])))
    layer = (z[None] >= top[1:, None, :]).sum(0).to(torch.float64)
    noise = 100.0 * torch.randn((1, 1, nz, nx), generator=g, device=dev, dtype=torch.float64)
    t = torch.exp(-0.5 * (torch.arange(-12, 13, device=dev, dtype=torch.float64) / 3.0) ** 2)
    t = t / t.sum()
    noise = F.conv2d(F.pad(noise, (12, 12, 0, 0), mode="replicate"), t.view(1, 1, 1, -1))
    noise = F.conv2d(F.pad(noise, (0, 0, 12, 12), mode="replicate"), t.view(1, 1, -1, 1))[0, 0]
    c = torch.clamp(1500.0 + 3000.0 * layer / 11.0 + noise, 1400.0, 4600.0)
    width = max(8, min(32, nx // 16))
    dx = torch.clamp(torch.maximum(width - x, x - (nx - 1 - width)), min=0.0)[None, :]
    dz = torch.clamp(z - (nz - 1 - width), min=0.0)
    gamma = torch.maximum(dx.expand(nz, nx), dz.expand(nz, nx)) / width
    return (1.0 / c).float().contiguous(), (gamma ** 2).float().contiguous()


def _param_shapes(widths=WIDTHS):
    """(cin, cout) of the network's layers in the order of its flat parameter vector."""
    c, n = list(widths), len(widths)
    s = [(3, c[0])] + [(c[0], c[0])] * 4
    for l in range(1, n):
        s += [(c[l - 1], c[l])] + [(c[l], c[l])] * 4
    for l in range(n - 2, -1, -1):
        s += [(c[l + 1], c[l]), (2 * c[l], c[l])] + [(c[l], c[l])] * 2
    s += [(3, c[0]), (2 * c[0], c[0])] + [(c[0], c[0])] * 2
    for l in range(1, n):
        s += [(c[l - 1], c[l]), (2 * c[l], c[l])] + [(c[l], c[l])] * 2
    for l in range(n - 2, -1, -1):
        s += [(c[l + 1], c[l]), (2 * c[l], c[l])] + [(c[l], c[l])] * 2
    return s + [(c[0], 2)]


def _params(case, g, dev):
    """Flat FP32 network parameters: the trained checkpoint's, or half-scale He-normal weights."""
    shapes = _param_shapes()
    n = sum(9 * i * o + o for i, o in shapes)
    if case["weights"] == "trained":
        return torch.from_numpy(np.fromfile(TRAINED, dtype=np.float32, count=n, offset=CKPT_HEADER_BYTES)).to(dev)
    out = []
    for i, o in shapes:
        out += [0.5 * math.sqrt(2.0 / (9 * i)) * torch.randn(9 * i * o, generator=g, device=dev),
                torch.zeros(o, device=dev)]
    return torch.cat(out)


def _inputs(case, seed):
    dev = _dev()
    g = torch.Generator(device=dev)
    g.manual_seed(int(seed))
    kind, nx, nz, nb = case["kind"], case["nx"], case["nz"], case["nrhs"]
    d = {}
    d["kappa"], d["gamma"] = _medium(case, g, dev)
    d["omegas"] = torch.tensor([2.0 * math.pi * f for f in _freqs(case)], dtype=torch.float32, device=dev)
    nfreq = len(_freqs(case))
    d["freq"] = np.minimum(np.arange(nb) * nfreq // nb, nfreq - 1).astype(np.int32)
    if kind in ("apply", "vcycle", "samples"):
        d["x"] = _cn(g, (nb, nz, nx), dev)
    if kind == "samples":
        d["iters"] = (np.arange(nb) % 10 + 1).astype(np.int32)
    if kind in ("precond", "loss_grad"):
        # residuals as a solver meets them: a few smooth waves and a rough part
        d["r"] = (_waves(g, nb, nz, nx, dev) + 0.3 * _cn(g, (nb, nz, nx), dev)).to(torch.complex64)
        d["params"] = _params(case, g, dev)
    if kind == "loss_grad":
        scale = case["hx"] * case["hz"]
        d["e"] = (scale * _waves(g, nb, nz, nx, dev)).to(torch.complex64)
    if kind == "residual":
        # a nearly converged iterate: H x agrees with the right-hand side to about 1e-5
        d["x"] = _waves(g, nb, nz, nx, dev)
        hx = torch.empty((nb, nz, nx), dtype=torch.complex64, device=dev)
        for j in range(nfreq):
            m = torch.from_numpy(np.flatnonzero(d["freq"] == j)).to(dev)
            hx[m] = _helmholtz(case, d, j)(d["x"][m]).to(torch.complex64)
        d["b"] = hx + 1e-5 * hx.abs().mean() * _cn(g, hx.shape, dev)
    if kind == "solve":
        # point sources on row 2, eight nodes apart, shifted by the seed
        pos = (4 + 8 * (np.arange(nb) % max(1, nx // 8)) + int(seed) % 5) % nx
        d["b"] = torch.zeros((nb, nz, nx), dtype=torch.complex64, device=dev)
        d["b"][torch.arange(nb, device=dev), 2, torch.from_numpy(pos).to(dev)] = 1.0 / (case["hx"] * case["hz"])
    if kind == "misfit":
        step = max(1, nx // nb)
        d["src"] = (2 * nx + (np.arange(nb) * step + int(seed) % step) % nx).astype(np.int32)
        d["rcv"] = (3 * nx + np.arange(case["nrcv"]) * (nx // case["nrcv"])).astype(np.int32)
        # observed data: the far field of a point source in 1.5 km/s water, with 10 % noise
        xs = torch.from_numpy(d["src"] % nx).to(dev) * case["hx"]
        xr = torch.from_numpy(d["rcv"] % nx).to(dev) * case["hx"]
        kr = d["omegas"].double()[:, None, None] / 1500.0 * (xr[None, :] - xs[:, None]).abs().clamp(min=case["hx"])
        far = torch.polar(0.25 * torch.sqrt(2.0 / (math.pi * kr)), -(kr + math.pi / 4))
        noise = _cn(g, far.shape, dev, torch.complex128)
        d["d_obs"] = (far * (1 + 0.1 * noise)).to(torch.complex64).contiguous()
    return d


def _waves(g, nb, nz, nx, dev, n=6):
    """Sums of n random plane waves of 8-20 points per wavelength (complex128 [nb][nz][nx])."""
    out = torch.zeros((nb, nz, nx), dtype=torch.complex128, device=dev)
    z = torch.arange(nz, device=dev, dtype=torch.float64)[None, :, None]
    x = torch.arange(nx, device=dev, dtype=torch.float64)[None, None, :]
    u = torch.rand((3, n, nb, 1, 1), generator=g, device=dev, dtype=torch.float64)
    for j in range(n):
        k = 2 * math.pi / (8 + 12 * u[0, j])
        a = 2 * math.pi * u[1, j]
        px = torch.polar(torch.ones_like(k * x), k * torch.cos(a) * x + 2 * math.pi * u[2, j])
        out += px * torch.polar(torch.ones_like(k * z), k * torch.sin(a) * z)
    return out


# ---- the measured pass ----------------------------------------------------------------

class _State:
    """Inputs, outputs and the library handles a user's program keeps."""

    def __init__(self, case, seed):
        from paper_2405_17696_gb300 import native
        self.native, self.case, self.ctx, self.net = native, case, None, None
        self.d = d = _inputs(case, seed)
        kind, nx, nz, nb = case["kind"], case["nx"], case["nz"], _nsys(case)
        dev = d["kappa"].device
        network = kind in ("precond", "loss_grad")
        if network:
            self.net = native.cnn_create(len(WIDTHS), WIDTHS)
            native.cnn_set_params(self.net, d["params"])
        opts = native.helm_default_opts(
            max_rhs=nb, max_iter=2000, precond=native.HELM_PC_CNN if network else native.HELM_PC_MG,
            stream=torch.cuda.current_stream(dev).cuda_stream)
        self.ctx = native.helm_setup(d["kappa"], d["gamma"], nx, nz, case["hx"], case["hz"], d["omegas"],
                                     net=self.net, opts=opts)
        field = lambda t: torch.empty((nb, nz, nx), dtype=t, device=dev)  # noqa: E731
        if kind in ("apply", "vcycle", "residual", "precond"):
            self.out = field(torch.complex64)
        elif kind == "samples":
            self.out = (field(torch.complex64), field(torch.complex64))
        elif kind == "solve":
            self.out = field(torch.complex128)
        elif kind == "misfit":
            self.out = torch.empty((nz, nx), dtype=torch.float32, device=dev)
        else:
            self.out = torch.empty(native.cnn_num_params(self.net), dtype=torch.float32, device=dev)

    def __del__(self):
        if self.ctx is not None:
            self.native.helm_destroy(self.ctx)
        if self.net is not None:
            self.native.cnn_destroy(self.net)


def prepare(case, seed):
    return _State(case, seed)


def run(s):
    n, c, d, nb = s.native, s.case, s.d, s.case["nrhs"]
    kind = c["kind"]
    if kind == "apply":
        n.helm_apply(s.ctx, d["x"], s.out, nb, d["freq"], c["op"])
        return s.out
    if kind == "vcycle":
        n.helm_vcycle(s.ctx, d["x"], None, s.out, nb, d["freq"])
        return s.out
    if kind == "residual":
        rel = n.helm_residual(s.ctx, d["b"], d["x"], s.out, nb, d["freq"])
        return {"r": s.out, "rel": rel}
    if kind == "samples":
        n.cnn_make_samples(s.ctx, d["x"], d["iters"], s.out[0], s.out[1], nb, d["freq"])
        return {"r": s.out[0], "e": s.out[1]}
    if kind == "solve":
        flags = n.HELM_SOLVE_ZERO_X0 | (n.HELM_SOLVE_ADJOINT if c["adjoint"] else 0)
        n.helm_solve(s.ctx, d["b"], s.out, nb, d["freq"], c["tol"], flags)
        # the wavefields in the precision of the data they are compared with
        return s.out.to(torch.complex64)
    if kind == "misfit":
        phi = n.fwi_misfit_grad(s.ctx, d["src"], d["rcv"], d["d_obs"], s.out, tol=c["tol"])
        return {"misfit": phi, "grad": s.out}
    if kind == "precond":
        n.cnn_precond_apply(s.ctx, d["r"], s.out, nb, d["freq"])
        return s.out
    loss = n.cnn_loss_grad(s.net, s.ctx, d["r"], d["e"], nb, d["freq"], s.out)
    return {"loss": loss, "grad": s.out}


def work(case):
    """Inputs read once, outputs written once; flops of the operator, cycle and network as defined."""
    kind, n, nb = case["kind"], case["nx"] * case["nz"], _nsys(case)
    pts = float(n * nb)
    vcyc = 180.0 * pts                                     # 4 sweeps, residual, transfers, coarser levels
    net = sum(2.0 * 9 * i * o / 4 ** l for (i, o), l in zip(_param_shapes(), _param_levels()))
    nsolver = 29
    solver = sum(2.0 * 9 * i * o / 4 ** l for (i, o), l in list(zip(_param_shapes(), _param_levels()))[-nsolver:])
    if kind == "apply":
        return {"bytes": 16 * pts + 8 * n, "flops": 22 * pts}
    if kind == "residual":
        return {"bytes": 32 * pts + 8 * n, "flops": 30 * pts}
    if kind == "vcycle":
        return {"bytes": 16 * pts + 8 * n, "flops": vcyc}
    if kind == "samples":
        return {"bytes": 24 * pts + 8 * n, "flops": 5.5 * (vcyc + 22 * pts + 2 * 8 * 5 * pts)}
    if kind in ("solve", "misfit"):
        # right-hand sides in, fields (and a gradient) out; the number of steps is the medium's
        return {"bytes": 24 * pts + 12 * n, "flops": vcyc}
    if kind == "precond":
        return {"bytes": 16 * pts + 8 * n, "flops": solver * pts + vcyc}
    return {"bytes": 16 * pts + 8 * n, "flops": 3 * (solver * pts + (net - solver) * n * len(_freqs(case)))}


def _param_levels():
    """Grid level each layer's output lies on, in the order of _param_shapes()."""
    n = len(WIDTHS)
    lv = [0] * 5
    for l in range(1, n):
        lv += [l] * 5
    for l in range(n - 2, -1, -1):
        lv += [l] * 4
    lv += [0] * 4
    for l in range(1, n):
        lv += [l] * 4
    for l in range(n - 2, -1, -1):
        lv += [l] * 4
    return lv + [0]


# ---- the same results in 64 bits, in plain torch ----------------------------------------

def _shift(u, dz, dx):
    """v(z, x) = u(z + dz, x + dx), zero outside."""
    nz, nx = u.shape[-2:]
    p = F.pad(torch.view_as_real(u), (0, 0, 1, 1, 1, 1))
    return torch.view_as_complex(p[..., 1 + dz:1 + dz + nz, 1 + dx:1 + dx + nx, :].contiguous())


def _five(coef, hx, hz):
    """u -> -Lap_h u - coef u."""
    ax, az = 1.0 / float(np.float32(hx)) ** 2, 1.0 / float(np.float32(hz)) ** 2

    def f(u):
        return ((2 * ax + 2 * az) * u - ax * (_shift(u, 0, -1) + _shift(u, 0, 1))
                - az * (_shift(u, -1, 0) + _shift(u, 1, 0)) - coef * u)
    f.diag = 2 * ax + 2 * az - coef
    return f


def _helmholtz(case, d, j, beta=None):
    """H of frequency j, or the shifted Laplacian with shift beta."""
    k, gam, w = d["kappa"].double(), d["gamma"].double(), float(d["omegas"][j])
    sig = gam if beta is None else gam + beta
    return _five(torch.complex(w * w * k * k, -w * w * k * k * sig), case["hx"], case["hz"])


def _restrict(r):
    t = (_shift(r, 0, -1) + 2 * r + _shift(r, 0, 1)) / 4
    t = (_shift(t, -1, 0) + 2 * t + _shift(t, 1, 0)) / 4
    return t[..., 1::2, 1::2].contiguous()


def _prolong(e):
    nz, nx = e.shape[-2:]
    f = torch.zeros(e.shape[:-2] + (2 * nz, 2 * nx), dtype=e.dtype, device=e.device)
    left = _shift(e, 0, -1)
    f[..., 1::2, 1::2], f[..., 1::2, 0::2] = e, 0.5 * (left + e)
    odd = f[..., 1::2, :]
    f[..., 0::2, :] = 0.5 * (odd + _shift(odd, -1, 0))
    return f


def _galerkin(fine, nz, nx, dev):
    """The nine-point operator R A (4 R^T), its coefficients read off nine coloured probes."""
    J = torch.arange(nz, device=dev)[:, None]
    I = torch.arange(nx, device=dev)[None, :]
    c = {}
    for a in range(3):
        for b in range(3):
            y = _restrict(fine(_prolong(((J % 3 == a) & (I % 3 == b)).to(torch.complex128))))
            for dz in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    m = ((J + dz) % 3 == a) & ((I + dx) % 3 == b)
                    c.setdefault((dz, dx), torch.zeros_like(y))
                    c[dz, dx] = torch.where(m, y, c[dz, dx])

    def f(u):
        return sum(c[k] * _shift(u, *k) for k in c)
    f.diag = c[0, 0]
    return f


def _levels(case, d, j, n=3):
    ops = [_helmholtz(case, d, j, beta=0.5)]
    for l in range(1, n):
        ops.append(_galerkin(ops[-1], case["nz"] >> l, case["nx"] >> l, d["kappa"].device))
    return ops


def _dot(a, b):
    return (a.conj() * b).sum((-2, -1))


def _gmres(A, M, b, steps):
    """Flexible GMRES from zero, steps[i] steps for right-hand side i (modified Gram-Schmidt)."""
    k, nb = max(steps), b.shape[0]
    V, Z, H = [], [], np.zeros((nb, k + 1, k), dtype=complex)
    beta = _dot(b, b).real.sqrt()
    safe = lambda t: torch.where(t > 0, t, torch.ones_like(t))[:, None, None]  # noqa: E731
    V.append(b / safe(beta))
    for j in range(k):
        Z.append(M(V[j]))
        w = A(Z[j])
        for i in range(j + 1):
            h = _dot(V[i], w)
            H[:, i, j] = h.cpu().numpy()
            w = w - h[:, None, None] * V[i]
        h = _dot(w, w).real.sqrt()
        H[:, j + 1, j] = h.cpu().numpy()
        V.append(w / safe(h))
    x = torch.zeros_like(b)
    y = np.zeros((nb, k), dtype=complex)
    for i, m in enumerate(steps):
        e1 = np.zeros(m + 1)
        e1[0] = float(beta[i])
        y[i, :m] = np.linalg.lstsq(H[i, :m + 1, :m], e1, rcond=None)[0]
    y = torch.from_numpy(y).to(b.device)
    for j in range(k):
        x += y[:, j, None, None] * Z[j]
    return x


def _vcycle(ops, f, l=0):
    if l == len(ops) - 1:
        return _gmres(ops[l], lambda v: v, f, [10] * f.shape[0])
    A = ops[l]
    u = 0.8 * f / A.diag
    u = u + 0.8 * (f - A(u)) / A.diag
    u = u + _prolong(_vcycle(ops, _restrict(f - A(u)), l + 1))
    for _ in range(2):
        u = u + 0.8 * (f - A(u)) / A.diag
    return u


class _Direct:
    """H x = b by block elimination over the columns (blocks of one grid column)."""

    def __init__(self, case, d, j):
        self.A = A = _helmholtz(case, d, j)
        nz, nx, dev = case["nz"], case["nx"], d["kappa"].device
        self.ax = 1.0 / float(np.float32(case["hx"])) ** 2
        az = 1.0 / float(np.float32(case["hz"])) ** 2
        off = -az * (torch.diag(torch.ones(nz - 1, device=dev, dtype=torch.complex128), 1)
                     + torch.diag(torch.ones(nz - 1, device=dev, dtype=torch.complex128), -1))
        self.S = []
        for i in range(nx):
            B = torch.diag(A.diag[:, i]) + off
            if i:
                B = B - self.ax ** 2 * self.S[-1]
            self.S.append(torch.linalg.inv(B))

    def once(self, b):
        c = b.permute(2, 1, 0)                              # [nx][nz][nrhs]
        y = [c[0]]
        for i in range(1, len(self.S)):
            y.append(c[i] + self.ax * (self.S[i - 1] @ y[-1]))
        x = [self.S[-1] @ y[-1]]
        for i in range(len(self.S) - 2, -1, -1):
            x.append(self.S[i] @ (y[i] + self.ax * x[-1]))
        return torch.stack(x[::-1]).permute(2, 1, 0).contiguous()

    def __call__(self, b):
        x = self.once(b)
        return x + self.once(b - self.A(x))


def _network(flat, xe, xs, zsel):
    """The encoder-solver network in 64 bits; xe [nfreq][3][nz][nx], xs [nb][3][nz][nx], zsel context per image."""
    shapes, at, n = _param_shapes(), [0, 0], len(WIDTHS)

    def conv(x, mode="same", relu=True, skip=None):
        i, o = shapes[at[0]]
        w = flat[at[1]:at[1] + 9 * i * o].view(o, 3, 3, i).permute(0, 3, 1, 2)
        b = flat[at[1] + 9 * i * o:at[1] + 9 * i * o + o]
        at[0], at[1] = at[0] + 1, at[1] + 9 * i * o + o
        if mode == "down":
            y = F.conv2d(F.pad(x, (0, 1, 0, 1)), w, b, stride=2)
        else:
            y = F.conv2d(F.interpolate(x, scale_factor=2, mode="nearest") if mode == "up" else x, w, b, padding=1)
        y = y if skip is None else y + skip
        return torch.relu(y) if relu else y

    def res(x):
        return conv(conv(x), skip=x)

    t = res(res(conv(xe)))
    e = [t]
    for l in range(1, n):
        t = res(res(conv(t, "down")))
        e.append(t)
    z = {n - 1: t}
    for l in range(n - 2, -1, -1):
        t = res(conv(torch.cat([conv(t, "up"), e[l]], 1)))
        z[l] = t
    t = res(conv(torch.cat([conv(xs), z[0][zsel]], 1)))
    s = [t]
    for l in range(1, n):
        t = res(conv(torch.cat([conv(t, "down"), z[l][zsel]], 1)))
        s.append(t)
    for l in range(n - 2, -1, -1):
        t = res(conv(torch.cat([conv(t, "up"), s[l]], 1)))
    return conv(t, relu=False)


def _net_error(case, d, flat):
    """e_net = hx hz rms(r) (out_0 + i out_1)."""
    r, k, gam = d["r"].to(torch.complex128), d["kappa"].double(), d["gamma"].double()
    hg = math.sqrt(case["hx"] * case["hz"])
    xe = torch.stack([torch.stack([1500.0 * k, gam, float(w) * hg * k]) for w in d["omegas"]])
    rms = (r.abs() ** 2).mean((-2, -1)).sqrt()[:, None, None]
    xs = torch.stack([r.real / rms, r.imag / rms, gam.expand(r.shape)], 1)
    o = _network(flat, xe, xs, torch.from_numpy(d["freq"].astype(np.int64)).to(r.device))
    return case["hx"] * case["hz"] * rms * torch.complex(o[:, 0], o[:, 1])


def exact(case, seed):
    kind, n, nb = case["kind"], case["nx"] * case["nz"], case["nrhs"]
    if kind == "loss_grad" and n * nb > 2e6:
        return None                                         # over twenty seconds in 64 bits
    d = _inputs(case, seed)
    dev = d["kappa"].device
    if kind == "loss_grad":
        flat = d["params"].double().requires_grad_(True)
        loss = ((_net_error(case, d, flat) - d["e"]).abs() ** 2).sum() / nb
        loss.backward()
        return {"loss": float(loss), "grad": flat.grad}
    if kind == "misfit":
        phi, grad = 0.0, torch.zeros((case["nz"], case["nx"]), dtype=torch.float64, device=dev)
        src, rcv = (torch.from_numpy(d[k].astype(np.int64)).to(dev) for k in ("src", "rcv"))
        for j, w in enumerate(d["omegas"].double()):
            solve = _Direct(case, d, j)
            b = torch.zeros((nb, n), dtype=torch.complex128, device=dev)
            b[torch.arange(nb, device=dev), src] = 1.0 / (case["hx"] * case["hz"])
            u = solve(b.view(nb, case["nz"], case["nx"]))
            r = u.view(nb, n)[:, rcv] - d["d_obs"][j]
            q = torch.zeros((nb, n), dtype=torch.complex128, device=dev)
            q[:, rcv] = r.conj()
            um = u * solve(q.view(u.shape))
            phi += float((r.abs() ** 2).sum())
            grad += 2 * float(w) ** 2 * (um.real + d["gamma"].double() * um.imag).sum(0)
        return {"misfit": phi, "grad": grad}
    outs = {}
    if kind == "precond":
        with torch.no_grad():
            e0 = torch.cat([_net_error(case, {**d, "r": d["r"][i:i + 4], "freq": d["freq"][i:i + 4]},
                                       d["params"].double()) for i in range(0, nb, 4)])
    for j in range(len(d["omegas"])):
        m = torch.from_numpy(np.flatnonzero(d["freq"] == j)).to(dev)
        if not len(m):
            continue
        if kind == "apply":
            got = {"": _helmholtz(case, d, j, 0.5 if case["op"] else None)(d["x"][m].to(torch.complex128))}
        elif kind == "residual":
            b = d["b"][m].to(torch.complex128)
            r = b - _helmholtz(case, d, j)(d["x"][m])
            got = {"r": r, "rel": (_dot(r, r).real / _dot(b, b).real).sqrt()}
        elif kind == "vcycle":
            got = {"": _vcycle(_levels(case, d, j), d["x"][m].to(torch.complex128))}
        elif kind == "solve":
            b = d["b"][m].to(torch.complex128)
            solve = _Direct(case, d, j)
            got = {"": solve(b.conj()).conj() if case["adjoint"] else solve(b)}
        elif kind == "samples":
            H, ops, x = _helmholtz(case, d, j), _levels(case, d, j), d["x"][m].to(torch.complex128)
            e = x - _gmres(H, lambda v: _vcycle(ops, v), H(x), [int(d["iters"][i]) for i in m.tolist()])
            got = {"r": H(e), "e": e}
        else:
            H, ops = _helmholtz(case, d, j), _levels(case, d, j)
            got = {"": e0[m] + _vcycle(ops, d["r"][m] - H(e0[m]))}
        for k, v in got.items():
            if k not in outs:
                outs[k] = torch.zeros((nb,) + v.shape[1:], dtype=v.dtype, device=dev)
            outs[k][m] = v
    if "rel" in outs:
        outs["rel"] = outs["rel"].cpu().numpy()
    return outs[""] if "" in outs else outs
