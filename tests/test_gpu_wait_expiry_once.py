"""A matcher wait that expires costs its seconds once, however many products the block's search
takes: with eight vertical offsets, and with a strip of sixteen products at one offset (both with
more sampled rows than the operand ring holds), the injected expiry ends the call within the sum
of one product's waits -- about two seconds each for a ring stage and for the products' end, and
about three for what is in flight; a second is allowed for the rest -- with every searched box
invalid, and the next call equals the oracle."""
import time

import numpy as np
import pytest

from oracle import oracle as orc
from paper_2604_07980_gb300 import workloads as wl
from tests.parity_util import compare_box_outputs, torch_frames

pytestmark = pytest.mark.gpu

SETS = {
    "offsets": dict(close_factor=1, far_dmax=27, close_dmax=27, dy_min=-4, dy_max=3),
    "wide strip": dict(far_side_px=4000, far_dmax=31),
}


@pytest.mark.parametrize("name", SETS)
def test_expiry_is_paid_once_per_call(name):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2604_07980_gb300 import binding as B
    W, H = 1400, 300
    w = wl.frame1080(seed=5400, W=W, H=H, n_boxes=1, side_range=(100, 200))
    f = w.frames[0]
    boxes = np.array([[40, 20, 1340, 280, 0]] if name == "wide strip" else
                     [[100, 40, 300, 200, 0], [500, 60, 640, 240, 0]], np.int32)
    params = {**w.params, **SETS[name]}
    ref = orc.match_frame(f.left, f.right, boxes, f.f_px, f.baseline_m, orc.Params(**params))
    L, R = torch_frames(w.frames)[0]
    b = torch.from_numpy(boxes).cuda()
    ctx = B.Context(params, 1, W, H, len(boxes))
    ctx.match_boxes(L, R, b, f.f_px, f.baseline_m)
    torch.cuda.synchronize()
    ctx.inject_wait_expiry()
    t0 = time.monotonic()
    got = ctx.match_boxes(L, R, b, f.f_px, f.baseline_m)
    torch.cuda.synchronize()
    seconds = time.monotonic() - t0
    assert ctx.stats()["error"] != 0
    assert 1.0 < seconds < 8.0, seconds
    assert (got["flags"].cpu().numpy() == 0).all() and torch.isnan(got["disp"]).all()
    got = ctx.match_boxes(L, R, b, f.f_px, f.baseline_m)
    torch.cuda.synchronize()
    assert ctx.stats()["error"] == 0
    compare_box_outputs({k: v.cpu().numpy() for k, v in got.items()}, ref, name)
    ctx.close()
