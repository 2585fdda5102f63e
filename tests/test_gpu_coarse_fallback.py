"""GPU parity of the coarsest-level solve on grids that no thread-block cluster holds (rows of more than 768 nodes, or
more than sixteen slabs), which take one block per right-hand side: even and odd numbers of columns."""
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


@pytest.mark.parametrize("nx,nz,k,nb", [
    (1600, 32, 10, 2),      # 800 x 16
    (1538, 16, 10, 3),      # 769 x 8
    (800, 272, 10, 1),      # 400 x 136
    (770, 400, 10, 2),      # 385 x 200
    (1554, 8, 4, 200),      # 777 x 4, more right-hand sides than SMs
])
def test_coarsest_solve_beyond_clusters(native, nx, nz, k, nb):
    dev = torch.device("cuda:0")
    h = 20.0
    kap, gam = media.kappa_of(media.layered_velocity(nx, nz, seed=5)), media.abl_gamma(nx, nz, 2 if nz < 32 else 8)
    om = np.asarray([2 * np.pi * 5.0], np.float32)
    f = media.complex_normal((nb, nz, nx), 7)
    opts = native.helm_default_opts(mg_levels=2, coarse_iters=k, max_rhs=nb, restart=1,
                                    stream=torch.cuda.current_stream(dev).cuda_stream)
    ctx = native.helm_setup(torch.from_numpy(kap).to(dev), torch.from_numpy(gam).to(dev), nx, nz, h, h,
                            torch.from_numpy(om).to(dev), opts=opts)
    try:
        u = torch.empty((nb, nz, nx), dtype=torch.complex64, device=dev)
        native.helm_vcycle(ctx, torch.from_numpy(f).to(dev), None, u, nb)
        got = u.cpu().numpy()
    finally:
        native.helm_destroy(ctx)
    pc = MG.VCyclePreconditioner(kap.astype(np.float64), gam.astype(np.float64), float(om[0]), h, h,
                                 MG.VCycleParams(levels=2, coarse_iters=k, jacobi_w=float(np.float32(0.8))))
    for b in sorted({0, nb - 1}):
        ref = pc(f[b].astype(np.complex128))
        # FP32 vectors: about 20 operations per node and level, as the V-cycle parity test allows
        assert np.abs(got[b] - ref).max() <= 2e-5 * np.abs(ref).max(), b
