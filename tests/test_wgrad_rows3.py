"""Weight-gradient plans whose three tap rows of a column shift come in one TMA box (same grid, tiles of one row, all taps
in one group: k_wgrad_tc.cu, rows3): the boxes' landing places, and the (tap, chunk) of every plane as the
producer lays them down and as the epilogue reads them.  No GPU is needed."""
import itertools

import pytest


@pytest.fixture(scope="module")
def n():
    from paper_2405_17696_gb300 import build
    build.build()
    from paper_2405_17696_gb300 import native
    return native


@pytest.mark.parametrize("c0,c1,npad", [(16, 0, 16), (16, 16, 16), (32, 0, 32), (32, 32, 32), (64, 0, 64)])
def test_three_row_boxes_fill_the_stage_once(n, c0, c1, npad):
    checked = 0
    for (h, w), nb, sms in itertools.product([(512, 1024), (256, 512), (7, 300), (1, 128), (2, 120), (37, 128)],
                                             (1, 16), (148, 152)):
        g = n.cnn_wgrad_plan(0, c0, c1, npad, h, w, nb, sms)
        if g["rows"] != 1 or g["ngroups"] != 1:
            continue
        checked += 1
        cx, cx0, plane = g["cx"], g["cx0"], g["plane"]
        assert plane == 16 * g["tw"] and 2 * g["tw"] <= 256 and cx <= 256   # a box row is a plane; three rows a box
        owner, total = {}, 0
        for sx in range(3):
            for first, count in ((0, cx0), (cx0, cx - cx0)):
                lo = sx * 3 * cx * plane + 3 * first * plane
                assert lo % 16 == 0 and lo + 3 * count * plane <= g["max_chunks"] * plane
                total += 3 * count * plane
                for chunk, dy in itertools.product(range(count), range(3)):   # rows vary faster than chunks
                    at = lo // plane + 3 * chunk + dy
                    assert at not in owner
                    owner[at] = (3 * dy + sx, first + chunk)
        # the transaction bytes of a tile
        assert total + g["gchunks"] * plane == (9 * cx + g["gchunks"]) * plane
        # the plane that the epilogue takes a row of the product from
        assert owner == {p: (p % 3 * 3 + p // 3 // cx, p // 3 % cx) for p in range(9 * cx)}
    assert checked or npad == 64
