"""GPU parity of the coarsest-level solve in thread-block clusters against the oracle: grids
whose slabs end inside a strip, an odd number of coarse columns, one to sixteen CTAs per
right-hand side, basis vectors that spill to global memory, short and long step counts, and
inactive right-hand sides' neighbours in a batch."""
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


@pytest.mark.parametrize("nx,nz,levels,k,nb", [
    (8, 8, 3, 10, 1),         # a 2 x 2 coarsest grid: GMRES ends before its ten steps
    (76, 48, 3, 10, 3),       # 19 coarse columns
    (64, 36, 3, 1, 2),        # one step; 9 coarse rows
    (64, 32, 3, 16, 5),       # the longest basis
    (104, 60, 3, 10, 40),     # 26 x 15
    (512, 256, 3, 10, 2),     # 128 x 64, a few CTAs per right-hand side
    (200, 96, 2, 10, 3),      # 100 x 48
    (512, 248, 2, 10, 2),     # 256 x 124: sixteen CTAs, the last with four rows of its slab
    (680, 344, 2, 10, 2),     # 340 x 172: basis vectors in global memory
    (1040, 64, 2, 10, 1),     # rows wider than a CTA of strips
])
def test_coarsest_solve_parity(native, nx, nz, levels, k, nb):
    dev = torch.device("cuda:0")
    h = 20.0
    c = media.layered_velocity(nx, nz, seed=5)
    kap, gam = media.kappa_of(c), media.abl_gamma(nx, nz, 2 if nx < 32 else 8)
    om = np.asarray([2 * np.pi * 4.0, 2 * np.pi * 6.0], np.float32)
    p = MG.VCycleParams(levels=levels, coarse_iters=k)
    f = media.complex_normal((nb, nz, nx), 7)
    fi = (np.arange(nb) % 2).astype(np.int32)
    if nb > 1:
        f[1] = 0.0            # a zero right-hand side: zero correction
    opts = native.helm_default_opts(mg_levels=levels, coarse_iters=k, max_rhs=nb,
                                    stream=torch.cuda.current_stream(dev).cuda_stream)
    ctx = native.helm_setup(torch.from_numpy(kap).to(dev), torch.from_numpy(gam).to(dev), nx, nz, h, h,
                            torch.from_numpy(om).to(dev), opts=opts)
    try:
        u = torch.empty((nb, nz, nx), dtype=torch.complex64, device=dev)
        native.helm_vcycle(ctx, torch.from_numpy(f).to(dev), None, u, nb, fi)
        got = u.cpu().numpy()
    finally:
        native.helm_destroy(ctx)
    for b in sorted({0, min(1, nb - 1), nb - 1}):
        ref = MG.VCyclePreconditioner(kap.astype(np.float64), gam.astype(np.float64), float(om[fi[b]]), h, h, p)(f[b])
        # FP32 vectors: about 20 operations per node and level, as the V-cycle parity test allows
        assert np.abs(got[b] - ref).max() <= 2e-5 * np.abs(ref).max() + (0.0 if f[b].any() else 1e-30), (b,)
