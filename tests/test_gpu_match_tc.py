"""The tensor-core matcher at the edges of its tiles: strips of 127 to 129 and 255 to 258
columns (one product, two products, more than one tile), odd first columns, points spread
so far apart that the strip has gaps, one to sixteen sampled rows (whole and partial ring
stages), few points, vertical search, strips that reach over every border of the plane.
Block records and every forward and backward cost equal the oracle's."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2604_07980_gb300 import workloads as wl
from tests.parity_util import compare_box_outputs, compare_debug, torch_frames

pytestmark = pytest.mark.gpu

W, H = 760, 90

# (box width, candidates): the sampled columns of a box of 16 s pixels span 15 s
SHAPES = [(16, 112), (16, 113), (16, 114), (64, 67), (64, 68), (64, 69), (48, 210), (48, 211), (48, 212), (48, 213),
          (3, 256), (320, 64), (640, 8), (704, 3), (720, 40)]


@pytest.mark.parametrize("width,nd", SHAPES)
@pytest.mark.parametrize("rows", [(16, 9, 4, 1), (13, 8, 3, 2)])
def test_strip_widths_and_rows_bit_exact(width, nd, rows):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2604_07980_gb300 import binding as B
    w = wl.multi_frame("frame1080", 9400 + 7 * width + nd, 1, W, H, 3, (20.0, 60.0), (0.5, 20.0), (0.5, 20.0))
    dmin = -3 if nd % 2 else 0
    ndy = 2 if nd <= 128 else 1
    params = dict(w.params, far_side_px=0, close_factor=1, grid_g=1, min_pts=1, agg_nmin=1, close_dmin=dmin,
                  close_dmax=dmin + nd - 1, far_dmin=dmin, far_dmax=dmin + nd - 1, dy_min=0, dy_max=ndy - 1,
                  max_occluders=0)
    boxes = []
    for i, h in enumerate(rows):
        for x0 in (4, 5, (W - width) // 2 + i, W - width - 4, W - width):
            y0 = (0, 3, 40, H - h)[(i + x0) % 4]
            boxes.append([min(max(x0, 0), W - width), y0, min(max(x0, 0), W - width) + width, y0 + h, 0])
    boxes = np.array(boxes, np.int32)
    fr = w.frames[0]
    ref = orc.match_frame(fr.left, fr.right, boxes, fr.f_px, fr.baseline_m, orc.Params(**params), debug=True)
    ctx = B.Context(params, 1, W, H, len(boxes))
    L, R = torch_frames([fr])[0]
    got = ctx.match_boxes(L, R, torch.from_numpy(boxes).cuda(), fr.f_px, fr.baseline_m, debug=True)
    torch.cuda.synchronize()
    where = f"width {width} candidates {nd} rows {rows}"
    compare_box_outputs({k: v.cpu().numpy() for k, v in got.items() if k != "debug"}, ref, where)
    compare_debug(got["debug"], ref, B.n_candidates(ctx.params), where)
    assert ctx.stats()["error"] == 0
    ctx.close()
