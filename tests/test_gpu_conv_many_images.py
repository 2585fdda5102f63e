"""The input gradient of an up layer for more images than a grid's second dimension has blocks: as in two halves."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb,hin,win", [(65535, 2, 2), (65536, 2, 2), (140000, 1, 3)])
def test_up_layer_input_gradient(nb, hin, win):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2405_17696_gb300 import build
    build.build()
    from paper_2405_17696_gb300 import native as n
    c, cout = 16, 16
    g = np.random.default_rng(nb)
    x = np.zeros((nb, hin, win, c), np.float32)
    w = (g.normal(size=(cout, 9, c)) / 12).astype(np.float32)
    gy = g.normal(size=(nb, 2 * hin, 2 * win, cout)).astype(np.float32)
    got = np.full(x.shape, np.nan, np.float32)
    n.cnn_conv3x3_backward(x, c, None, 0, 0, nb, hin, win, w, cout, 2, gy, got)
    half = nb // 2
    for i, j in ((0, half), (half, nb)):
        want = np.full(x[i:j].shape, np.nan, np.float32)
        n.cnn_conv3x3_backward(x[i:j], c, None, 0, 0, j - i, hin, win, w, cout, 2, np.ascontiguousarray(gy[i:j]), want)
        assert np.isfinite(want).all() and np.array_equal(got[i:j], want)
