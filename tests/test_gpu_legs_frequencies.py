"""The coarse V-cycle legs repeat a tile's march for each frequency among a block's four right-hand sides, in the
same shared-memory rings.  A batch whose frequencies alternate within every block equals, bit for bit, the same
right-hand sides in batches of one frequency; segments of 64 rows and of 50 (2 modulo 8), more than one of them, so
that a march's look-ahead would reach rows of the next segment."""
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


@pytest.mark.parametrize("nx,nz,nb", [(512, 256, 190), (512, 200, 190)])
def test_mixed_frequencies_equal_single_ones(native, nx, nz, nb):
    dev = torch.device("cuda:0")
    kap = torch.from_numpy(media.kappa_of(media.layered_velocity(nx, nz, seed=6))).to(dev)
    gam = torch.from_numpy(media.abl_gamma(nx, nz, 16)).to(dev)
    om = torch.tensor([2 * np.pi * f for f in (3.0, 4.5, 6.0)], dtype=torch.float32, device=dev)
    opts = native.helm_default_opts(max_rhs=nb, restart=1, stream=torch.cuda.current_stream(dev).cuda_stream)
    ctx = native.helm_setup(kap, gam, nx, nz, 20.0, 20.0, om, opts=opts)
    try:
        f = torch.from_numpy(media.complex_normal((nb, nz, nx), 9)).to(dev)
        fi = (np.arange(nb) % 3).astype(np.int32)
        u, one = torch.empty_like(f), torch.empty_like(f)
        native.helm_vcycle(ctx, f, None, u, nb, fi)
        assert torch.isfinite(torch.view_as_real(u)).all()
        for k in range(3):
            native.helm_vcycle(ctx, f, None, one, nb, np.full(nb, k, np.int32))
            rows = torch.from_numpy(np.nonzero(fi == k)[0]).to(dev)
            assert torch.equal(torch.view_as_real(u[rows]).view(torch.int32), torch.view_as_real(one[rows]).view(torch.int32))
    finally:
        native.helm_destroy(ctx)
