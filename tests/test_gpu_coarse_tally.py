"""Bytes that the profiler books for the coarsest solve: its input and output where a cluster holds the basis on chip,
the basis too where one block per right-hand side keeps it in memory."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_2405_17696_gb300 import media  # noqa: E402


@pytest.mark.parametrize("nx,nz,k,nb,per_node", [
    (80, 64, 10, 3, 16),                                # 40 x 32, in a cluster
    (1600, 32, 4, 2, 8 * (4 * 4 + 5 * 4 + 2)),          # 800 x 16, in no cluster
])
def test_bytes_of_the_coarsest_solve(nx, nz, k, nb, per_node):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_17696_gb300 import build
    build.build()
    from paper_2405_17696_gb300 import native as n
    dev = torch.device("cuda:0")
    opts = n.helm_default_opts(mg_levels=2, coarse_iters=k, max_rhs=nb, restart=1,
                               stream=torch.cuda.current_stream(dev).cuda_stream)
    ctx = n.helm_setup(torch.from_numpy(media.kappa_of(media.layered_velocity(nx, nz, seed=1))).to(dev),
                       torch.from_numpy(media.abl_gamma(nx, nz, 8)).to(dev), nx, nz, 20.0, 20.0,
                       torch.tensor([2 * np.pi * 4.0], dtype=torch.float32, device=dev), opts=opts)
    try:
        f = torch.from_numpy(media.complex_normal((nb, nz, nx), 2)).to(dev)
        u = torch.empty_like(f)
        n.helm_profile_enable(ctx, True)
        n.helm_vcycle(ctx, f, None, u, nb)
        _, launches, nbytes = n.helm_profile_read(ctx)["coarse_gmres"]
        assert launches == 1 and nbytes == per_node * (nx // 2) * (nz // 2) * nb
    finally:
        n.helm_destroy(ctx)
