"""An up layer whose output has more than 2^31 pixels (image indices beyond 32 bits): small whole numbers, exact in BF16,
so that the outputs are whole numbers too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def test_up_layer_beyond_32_bit_pixels():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if torch.cuda.mem_get_info()[0] < 130e9:
        pytest.skip("needs 130 GB of free device memory")
    from paper_2405_17696_gb300 import build
    build.build()
    from paper_2405_17696_gb300 import native as n
    h = w = 23172
    assert 4 * h * w > 2 ** 31
    g = torch.Generator(device="cuda").manual_seed(3)
    x = torch.randint(0, 3, (h, w), generator=g, device="cuda").float()
    wt = np.array([[2, -1, 0], [1, 2, -2], [0, 1, 1]], np.float32)
    y = torch.full((2 * h, 2 * w), float("nan"), device="cuda")
    n.cnn_conv3x3(x, 1, None, 0, 0, 1, h, w, wt.reshape(1, 9, 1), np.array([3.0], np.float32), 1, None, 2, 0, y)
    for row in (0, 1, 30001, 2 ** 31 // (2 * w) - 1, 2 ** 31 // (2 * w) + 1, 2 * h - 1):
        want = torch.full((2 * w,), 3.0, device="cuda")
        for dy in (-1, 0, 1):
            if not 0 <= row + dy < 2 * h:
                continue
            fine = torch.nn.functional.pad(x[(row + dy) // 2].repeat_interleave(2), (1, 1))
            for dx in (-1, 0, 1):
                want += float(wt[dy + 1, dx + 1]) * fine[1 + dx:1 + dx + 2 * w]
        assert torch.equal(y[row], want), row
