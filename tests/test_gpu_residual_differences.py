"""The FP64 residual of smooth iterates keeps the differences of neighbours: against extended precision it is no
further off than the operator in the order it is written, at 160 and 640 points per wavelength (where five terms of a
node in one product cancel: ten to a hundred times that)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def native():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_17696_gb300 import build
    build.build()
    from paper_2405_17696_gb300 import native as n
    return n


@pytest.mark.parametrize("ppw,hx,hz,nb", [(160, 10.0, 8.0, 1), (160, 10.0, 13.0, 3), (640, 10.0, 10.0, 2)])
def test_residual_error_no_larger_than_in_written_order(native, ppw, hx, hz, nb):
    dev = torch.device("cuda:0")
    nx, nz, c0 = 64, 76, 2000.0
    kap = np.full((nz, nx), 1.0 / c0, np.float32)
    gam = np.full((nz, nx), 0.05, np.float32)
    om = np.float32(2 * np.pi * c0 / (ppw * max(hx, hz)))
    k = float(om) / c0
    X, Z = np.meshgrid(np.arange(nx) * hx, np.arange(nz) * hz)
    x = np.stack([np.exp(1j * (k * (0.8 * X + 0.6 * Z) + 0.7 + b)) * (1.2345 + b) for b in range(nb)])

    def parts(real):                    # H x in the order the operator is written, (re, im), in the type `real`
        re, im = x.real.astype(real), x.imag.astype(real)
        ax, az = real(1.0) / (real(hx) * real(hx)), real(1.0) / (real(hz) * real(hz))
        s = real(om) * real(om) * (kap.astype(real) * kap.astype(real))
        g = s * gam.astype(real)

        def lap(v):
            p = np.pad(v, ((0, 0), (1, 1), (1, 1)))
            return (ax * (2 * v - p[:, 1:-1, :-2] - p[:, 1:-1, 2:]) + az * (2 * v - p[:, :-2, 1:-1] - p[:, 2:, 1:-1]))
        return lap(re) - (s * re + g * im), lap(im) - (s * im - g * re)

    exact, written = parts(np.longdouble), parts(np.float64)
    assert np.finfo(np.longdouble).nmant > 60
    b = exact[0].astype(np.float32) + 1j * exact[1].astype(np.float32)
    opts = native.helm_default_opts(max_rhs=nb, mg_levels=2, restart=1, stream=torch.cuda.current_stream(dev).cuda_stream)
    ctx = native.helm_setup(torch.from_numpy(kap).to(dev), torch.from_numpy(gam).to(dev), nx, nz, hx, hz,
                            torch.tensor([om], dtype=torch.float32, device=dev), opts=opts)
    try:
        r = torch.empty((nb, nz, nx), dtype=torch.complex64, device=dev)
        native.helm_residual(ctx, torch.from_numpy(b.astype(np.complex64)).to(dev), torch.from_numpy(x).to(dev), r, nb)
        got = r.cpu().numpy()
    finally:
        native.helm_destroy(ctx)

    def rms(v):                         # (the zeros beyond the grid make the outermost nodes large)
        return float(np.sqrt(np.mean(v[:, 1:-1, 1:-1].astype(np.float64) ** 2)))

    for part, bp, e, w in ((got.real, b.real, exact[0], written[0]), (got.imag, b.imag, exact[1], written[1])):
        want = bp.astype(np.longdouble) - e
        # twice the written order's error, the coefficient's own rounding, and the result's, stored in FP32
        bound = 2 * rms(w.astype(np.longdouble) - e) + 2.0 ** -51 * rms(e) + 2.0 ** -24 * rms(want)
        assert rms(part.astype(np.longdouble) - want) <= bound
