"""GPU parity of the fused V-cycle legs against the oracle, where a strip of columns or a
segment of rows ends: strips one pair short of and past their 29 and 30 useful pairs, heights
around a segment, the smallest grids, deeper hierarchies, and against the separate sweep and
transfer kernels (which an initial guess of zeros takes)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from oracle import multigrid as MG  # noqa: E402
from paper_2405_17696_gb300 import media  # noqa: E402


@pytest.fixture(scope="module")
def native():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_17696_gb300 import build
    build.build()
    from paper_2405_17696_gb300 import native as n
    return n


@pytest.mark.parametrize("nx,nz,levels,nb,hz", [
    (4, 4, 2, 1, 20.0),           # one pair of coarse nodes
    (8, 60, 2, 3, 20.0),
    (56, 32, 2, 2, 20.0), (60, 34, 2, 2, 20.0), (64, 66, 2, 2, 24.0),      # 28, 30 and 32 pairs
    (116, 64, 3, 2, 20.0), (120, 68, 3, 2, 20.0), (124, 136, 3, 5, 16.0),  # 58, 60 and 62 pairs
    (352, 176, 4, 2, 20.0),
    (160, 128, 3, 70, 20.0),      # more right-hand sides than warps of a block
])
def test_legs_parity(native, nx, nz, levels, nb, hz):
    dev = torch.device("cuda:0")
    h = 20.0
    kap, gam = media.kappa_of(media.layered_velocity(nx, nz, seed=3)), media.abl_gamma(nx, nz, min(8, nx // 4))
    om = np.asarray([2 * np.pi * 4.0, 2 * np.pi * 7.0], np.float32)
    f = media.complex_normal((nb, nz, nx), 11)
    fi = (np.arange(nb) % 2).astype(np.int32)
    p = MG.VCycleParams(levels=levels, jacobi_w=float(np.float32(0.8)))
    opts = native.helm_default_opts(mg_levels=levels, max_rhs=nb, stream=torch.cuda.current_stream(dev).cuda_stream)
    ctx = native.helm_setup(torch.from_numpy(kap).to(dev), torch.from_numpy(gam).to(dev), nx, nz, h, hz,
                            torch.from_numpy(om).to(dev), opts=opts)
    try:
        fd = torch.from_numpy(f).to(dev)
        u, v = torch.empty_like(fd), torch.empty_like(fd)
        native.helm_vcycle(ctx, fd, None, u, nb, fi)
        native.helm_vcycle(ctx, fd, torch.zeros_like(fd), v, nb, fi)
        got, sep = u.cpu().numpy(), v.cpu().numpy()
    finally:
        native.helm_destroy(ctx)
    # the fused legs take the separate kernels' operations in the same order
    assert np.array_equal(got, sep)
    for b in sorted({0, nb // 2, nb - 1}):
        pc = MG.VCyclePreconditioner(kap.astype(np.float64), gam.astype(np.float64), float(om[fi[b]]), h, hz, p)
        ref = pc(f[b].astype(np.complex128))
        # complex64 arithmetic through four sweeps a level: a few units of 2^-23 of the largest value each
        assert np.abs(got[b] - ref).max() <= 2e-5 * np.abs(ref).max(), b
