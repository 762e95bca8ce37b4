"""The offset search at the edges of its two kernels: pixel segments narrower and wider than
three ranges (where the choice lies), one and more segments of 2048 pixels, steps of 64 pixels
filled exactly and by one pixel, regions at and beyond the image borders, negative and single
disparities, offsets that leave the image, and the three kinds of census window; counts equal
the oracle's."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2604_07980_gb300 import workloads as wl

CASES = [
    # W, H, roi, dmin, dmax, delta range, window
    (300, 24, (30, 4, 221, 20), 0, 63, (-2, 2), (9, 7)),      # 191 < 3 * 64: a thread per pixel
    (300, 24, (30, 4, 222, 20), 0, 63, (-2, 2), (9, 7)),      # 192 = 3 * 64: the band
    (260, 20, (0, 0, 260, 20), -7, 24, (-3, 1), (7, 7)),      # whole image, negative disparities
    (260, 20, (-9, -5, 300, 40), 0, 0, (0, 0), (5, 5)),       # one disparity, region beyond the image
    (2400, 14, (100, 3, 2280, 12), 0, 40, (-1, 1), (9, 7)),   # a full segment and a short one
    (2100, 12, (26, 2, 2074, 11), 3, 35, (0, 12), (11, 5)),   # exactly one segment; rows leave the image
    (700, 16, (50, 2, 690, 15), 0, 200, (-1, 0), (3, 15)),    # a long range
]


@pytest.mark.gpu
@pytest.mark.parametrize("case", range(len(CASES)))
def test_offset_counts_equal_oracle(case):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2604_07980_gb300 import binding as B
    W, H, roi, dmin, dmax, (lo, hi), win = CASES[case]
    rng = np.random.default_rng(3300 + case)
    big = np.clip(np.rint(wl.texture(rng, H + 4, W + 20)), 0, 255).astype(np.uint8)
    L = big[2:2 + H, :W].copy()
    R = big[3:3 + H, 11:11 + W].copy()
    R[:, W // 2:] = rng.integers(0, 256, (H, W - W // 2), dtype=np.uint8)
    ref_best, ref_counts = orc.auto_rect(L, R, roi, dmin, dmax, lo, hi, 1, win_w=win[0], win_h=win[1])
    delta, counts = B.auto_rect(torch.from_numpy(L).cuda(), torch.from_numpy(R).cuda(), roi, dmin, dmax, lo, hi, 1,
                                params=dict(win_w=win[0], win_h=win[1]))
    torch.cuda.synchronize()
    assert np.array_equal(counts.cpu().numpy(), ref_counts)
    assert int(delta.item()) == ref_best
