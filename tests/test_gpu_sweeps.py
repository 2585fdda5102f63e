"""The V-cycle by a kernel per sweep and transfer, which the default cycle's one pass per leg stands for: the same
bits on every level, and the same bits whatever block shapes helm_autotune records for the sweeps."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2405_17696_gb300 import media  # noqa: E402


@pytest.fixture(scope="module")
def native():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_17696_gb300 import build
    build.build()
    from paper_2405_17696_gb300 import native as n
    return n


def _context(native, nx, nz, nb, **opts):
    dev = torch.device("cuda:0")
    kap = torch.from_numpy(media.kappa_of(media.layered_velocity(nx, nz, seed=8))).to(dev)
    gam = torch.from_numpy(media.abl_gamma(nx, nz, min(8, nx // 4))).to(dev)
    om = torch.tensor([2 * np.pi * f for f in (3.0, 5.0, 6.0)], dtype=torch.float32, device=dev)
    o = native.helm_default_opts(max_rhs=nb, stream=torch.cuda.current_stream(dev).cuda_stream, **opts)
    return native.helm_setup(kap, gam, nx, nz, 20.0, 20.0, om, opts=o)


def _bits(x):
    return torch.view_as_real(x).view(torch.int32)


@pytest.mark.parametrize("nx,nz,levels,nb", [
    (8, 12, 3, 1),              # a pair of columns on the coarser level
    (120, 68, 3, 5),            # 60 and 30 pairs of columns
    (256, 176, 4, 9),           # legs on two coarse levels
    (512, 256, 3, 190),         # 64-row segments on the coarse level
])
def test_legs_equal_separate_kernels_on_every_level(native, nx, nz, levels, nb):
    ctx = _context(native, nx, nz, nb, mg_levels=levels, restart=1)
    try:
        f = torch.from_numpy(media.complex_normal((nb, nz, nx), 3)).cuda()
        fi = (np.arange(nb) % 3).astype(np.int32)
        u, v = torch.empty_like(f), torch.empty_like(f)
        native.helm_vcycle(ctx, f, None, u, nb, fi)
        native.helm_set_legs(ctx, False)
        native.helm_vcycle(ctx, f, None, v, nb, fi)
        assert torch.isfinite(torch.view_as_real(v)).all()
        assert torch.equal(_bits(u), _bits(v))
    finally:
        native.helm_destroy(ctx)


@pytest.mark.parametrize("opts,legs", [(dict(pre=1, post=1), True), (dict(pre=2, post=1), True), (dict(), False)])
def test_tuned_sweeps_keep_the_bits(native, opts, legs):
    nx, nz, nb = 192, 96, 3
    native.helm_autotune_reset()
    ctx = _context(native, nx, nz, nb, mg_levels=3, **opts)
    try:
        native.helm_set_legs(ctx, legs)
        f = torch.from_numpy(media.complex_normal((nb, nz, nx), 4)).cuda()
        fi = np.array([0, 1, 2], np.int32)
        u, x = [], []
        for tuned in (False, True):
            if tuned:
                assert native.helm_autotune(ctx, nb) >= 2       # the fine sweep and at least one coarse level
            u.append(torch.empty_like(f))
            native.helm_vcycle(ctx, f, None, u[-1], nb, fi)
            x.append(torch.zeros(f.shape, dtype=torch.complex128, device="cuda"))
            native.helm_solve(ctx, f, x[-1], nb, fi, 1e-4, native.HELM_SOLVE_ZERO_X0)
        assert torch.equal(_bits(u[0]), _bits(u[1])) and torch.equal(x[0], x[1])
    finally:
        native.helm_destroy(ctx)
        native.helm_autotune_reset()
