"""The same-grid convolution with adjacent row accumulators (k_conv_tma.cu, mode 5), which a
default launch takes where it needs fewer tensor-core cycles: its schedule on the CPU, run from the
library's own plans, and on the GPU its results against the plain kernel's, which sums the same
products in the same order, so that they are equal bit for bit."""
import itertools

import numpy as np
import pytest


@pytest.fixture(scope="module")
def n():
    from paper_2405_17696_gb300 import build
    build.build()
    from paper_2405_17696_gb300 import native
    return native


def test_schedule_stays_in_bounds_and_keeps_the_order(n):
    """Every operand read lies in its stage, every accumulator column in its buffer, and each
    output row takes its nine taps once, in the plain kernel's order."""
    checked = 0
    for (H, W), c0, c1, npad in itertools.product(
            [(1, 126), (2, 120), (3, 127), (7, 300), (8, 114), (9, 252), (33, 129), (37, 113), (256, 512), (512, 1024)],
            (16, 64), (0, 32), (16, 32, 64, 96, 128)):
        g = n.cnn_conv_plan(0, c0, c1, npad, H, W, 2, narrow=6)
        if g is None or g["mode"] != 5:
            assert npad >= 64 or H < 4 or (W + (W + 125) // 126 - 1) // ((W + 125) // 126) < 80, (H, W, npad, g)
            continue
        checked += 1
        R, pw, plane, wofs = g["rows"], g["pw"], g["plane"], g["pstride"]
        assert pw == g["tw"] + 2 <= 128 and 3 * npad <= 256 and R * npad <= 256
        assert g["nbuf"] * R * npad <= g["tmem_cols"] <= 512
        assert g["ns"] >= 2 and g["ns"] * g["stage"] + 256 * 32 + 2048 <= 227 * 1024
        assert wofs + g["wbytes"] <= g["stage"] and g["wbytes"] == 9 * 2 * npad * 16
        taps = [[] for _ in range(R)]
        for b in range(R + 2):
            t0, t1 = (0 if b < R else b - R + 1), (b if b < 2 else 2)
            col, ncol = (R - 1 - b + t0) * npad, (t1 - t0 + 1) * npad
            assert 0 <= col and col + ncol <= R * npad
            for dx in range(3):
                for h in (0, 1):
                    a = h * plane + (b * pw + dx) * 16
                    assert a + 128 * 16 <= g["stage"]
                    w = (dx * 6 + h * 3) * npad * 16 + t0 * npad * 16
                    assert w + ncol * 16 <= (dx * 6 + h * 3 + 3) * npad * 16 <= g["wbytes"]
                for t in range(t0, t1 + 1):
                    r = R - 1 - (col // npad + t - t0)      # output row of the tap row's columns
                    assert r == b - t
                    taps[r].append((t, dx))
        assert all(x == [(t, dx) for t in range(3) for dx in range(3)] for x in taps)
    assert checked > 30


@pytest.mark.gpu
@pytest.mark.parametrize("c0,c1,bcast,cout,hin,win,nb,res,relu", [
    (16, 0, 0, 16, 2, 126, 1, 0, 1),        # two rows, a full tile of 126
    (16, 16, 0, 16, 9, 250, 3, 0, 0),       # two groups, ragged rows, two column tiles
    (32, 16, 1, 32, 37, 113, 2, 1, 1),      # batch-shared second input, residual
    (16, 0, 0, 2, 8, 114, 2, 0, 0),         # output layer, FP32, 2 of 16 channels stored
    (64, 0, 0, 64, 40, 252, 2, 1, 1),       # 64 channels, N up to 192
    (16, 0, 0, 16, 512, 1024, 6, 1, 1),     # several tiles per CTA, both accumulator buffers
    (32, 32, 0, 32, 256, 500, 8, 0, 1),
])
def test_equals_the_plain_kernel(n, c0, c1, bcast, cout, hin, win, nb, res, relu):
    torch = pytest.importorskip("torch")
    npad = 16 if cout <= 16 else 32 * -(-cout // 32)
    assert n.cnn_conv_plan(0, c0, c1, npad, hin, win, nb, narrow=6)["mode"] == 5
    g = torch.Generator().manual_seed(c0 + hin)
    x0 = torch.randn((nb, hin, win, c0), generator=g).cuda()
    x1 = torch.randn(((1 if bcast else nb), hin, win, c1), generator=g).cuda() if c1 else None
    r = torch.randn((nb, hin, win, cout), generator=g).cuda() if res else None
    w = (torch.randn((cout, 9, c0 + c1), generator=g) / np.sqrt(9 * (c0 + c1))).numpy()
    b = torch.randn((cout,), generator=g).numpy()
    out = []
    for cap in (0, 254):                    # a height limit that limits nothing takes the plain kernel
        y = torch.full((nb, hin, win, cout), float("nan"), device="cuda")
        n.cnn_set_conv_tiling(cap)
        try:
            n.cnn_conv3x3(x0, c0, x1, c1, bcast, nb, hin, win, w, b, cout, r, 0, relu, y)
        finally:
            n.cnn_set_conv_tiling(0)
        out.append(y.cpu())
    assert torch.isfinite(out[0]).all()
    assert torch.equal(out[0], out[1])
