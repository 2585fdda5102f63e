"""cnn_precond_apply and cnn_make_samples work on the caller's device arrays as they are and stage others:
host arrays, arrays off 16 bytes and overlapping ones give the same results, and inputs stay as they were."""
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


@pytest.mark.parametrize("nx,nz,cap,nb", [(64, 32, 3, 5), (32, 64, 2, 1)])
def test_results_do_not_depend_on_where_the_arrays_are(native, nx, nz, cap, nb):
    dev = torch.device("cuda:0")
    kap = torch.from_numpy(media.kappa_of(media.layered_velocity(nx, nz, seed=2))).to(dev)
    gam = torch.from_numpy(media.abl_gamma(nx, nz, 4)).to(dev)
    om = torch.tensor([2 * np.pi * 5.0], dtype=torch.float32, device=dev)
    opts = native.helm_default_opts(max_rhs=cap, restart=1, precond=native.HELM_PC_CNN,
                                    stream=torch.cuda.current_stream(dev).cuda_stream)
    net = native.cnn_create(2, (16, 32), 5)
    ctx = native.helm_setup(kap, gam, nx, nz, 20.0, 20.0, om, opts=opts, net=net)
    try:
        r0 = torch.from_numpy(media.complex_normal((nb, nz, nx), 3)).to(dev)
        r = r0.clone()
        want = torch.empty_like(r)
        native.cnn_precond_apply(ctx, r, want, nb)
        assert torch.equal(r, r0) and torch.isfinite(torch.view_as_real(want)).all()
        host = np.zeros((nb, nz, nx), np.complex64)
        native.cnn_precond_apply(ctx, r0.cpu().numpy(), host, nb)
        assert np.array_equal(host, want.cpu().numpy())
        same = r0.clone()
        native.cnn_precond_apply(ctx, same, same, nb)                    # in place
        assert torch.equal(same, want)
        buf = torch.zeros(2 * nb * nz * nx + 2, dtype=torch.complex64, device=dev)
        off_r, off_e = buf[1:1 + nb * nz * nx].view(nb, nz, nx), buf[nb * nz * nx + 1:-1].view(nb, nz, nx)
        off_r.copy_(r0)                                                  # 8 bytes off a boundary
        native.cnn_precond_apply(ctx, off_r, off_e, nb)
        assert torch.equal(off_e, want) and torch.equal(off_r, r0)

        m = min(nb, cap)
        x0, iters = r0[:m].clone(), [1] * m
        x = x0.clone()
        rs, es = torch.empty_like(x), torch.empty_like(x)
        native.cnn_make_samples(ctx, x, iters, rs, es, m)
        assert torch.equal(x, x0)
        hr, he = np.zeros((m, nz, nx), np.complex64), np.zeros((m, nz, nx), np.complex64)
        native.cnn_make_samples(ctx, x0.cpu().numpy(), iters, hr, he, m)
        assert np.array_equal(hr, rs.cpu().numpy()) and np.array_equal(he, es.cpu().numpy())
        xa, ra = x0.clone(), torch.empty_like(x)
        native.cnn_make_samples(ctx, xa, iters, ra, xa, m)               # e over x
        assert torch.equal(ra, rs) and torch.equal(xa, es)
    finally:
        native.helm_destroy(ctx)
        native.cnn_destroy(net)
