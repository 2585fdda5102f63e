"""helm_apply takes the operator on node pairs for large batches and by nodes otherwise, with the same rounded
operations: a batch on one side of the line equals its fields applied one by one on the other, bit for bit."""
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


@pytest.mark.parametrize("nx,nz,nb", [(512, 256, 12), (512, 256, 11), (328, 132, 40), (8, 1024, 200)])
def test_batch_equals_single_fields(native, nx, nz, nb):
    dev = torch.device("cuda:0")
    kap = torch.from_numpy(media.kappa_of(media.layered_velocity(nx, nz, seed=4))).to(dev)
    gam = torch.from_numpy(media.abl_gamma(nx, nz, min(8, nx // 4))).to(dev)
    om = torch.tensor([20.0, 41.0], dtype=torch.float32, device=dev)
    opts = native.helm_default_opts(max_rhs=nb, mg_levels=2, stream=torch.cuda.current_stream(dev).cuda_stream)
    ctx = native.helm_setup(kap, gam, nx, nz, 20.0, 16.0, om, opts=opts)
    try:
        x = torch.from_numpy(media.complex_normal((nb, nz, nx), 5)).to(dev)
        f = (np.arange(nb) % 2).astype(np.int32)
        y, one = torch.empty_like(x), torch.empty_like(x)
        native.helm_apply(ctx, x, y, nb, f)
        for b in range(nb):
            native.helm_apply(ctx, x[b:b + 1], one[b:b + 1], 1, f[b:b + 1])
        assert torch.isfinite(torch.view_as_real(y)).all()
        assert torch.equal(torch.view_as_real(y).view(torch.int32), torch.view_as_real(one).view(torch.int32))
    finally:
        native.helm_destroy(ctx)
