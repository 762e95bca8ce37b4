"""A host batch is copied in one part or in up to four, by its image bytes: at 3840x2160 one
part below 4 frames, two from 4, three from 7, four from 9.  Results equal the device batch's
bit for bit, also with a frame without boxes and with none at all, copying and mapped."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("frames", [1, 3, 4, 7, 9])
def test_host_parts_equal_device_batch(frames):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2604_07980_gb300 import binding as B
    W, H = 3840, 2160
    rng = np.random.default_rng(frames)
    left = torch.randint(0, 256, (frames, H, W), dtype=torch.uint8, device="cuda")
    images = torch.stack([left, torch.roll(left, -8, 2)], 1)
    rows = []
    for f in range(frames):
        for _ in range(0 if f == frames // 2 and frames > 1 else 5):
            w, h = int(rng.integers(12, 500)), int(rng.integers(12, 500))
            x, y = int(rng.integers(0, W - w)), int(rng.integers(0, H - h))
            rows.append([x, y, x + w, y + h, f])
    boxes = np.array(rows, np.int32)
    ctx = B.Context(None, frames, W, H, len(boxes))
    batch = B.DeviceBatch([(im[0], im[1]) for im in images], boxes, [(2000.0, 0.3)] * frames)
    ref = {k: v.cpu().numpy() for k, v in ctx.match_batch(batch).items()}
    assert (ref["flags"] & 1).any()
    host = images.cpu().pin_memory().numpy()
    for mapped in (False, True):
        got = ctx.match_batch_host_packed(host, boxes, 2000.0, 0.3, mapped=mapped)
        for k in ("disp", "depth", "flags"):
            assert got[k].tobytes() == ref[k].tobytes(), (mapped, k)
        none = ctx.match_batch_host_packed(host, boxes[:0], 2000.0, 0.3, mapped=mapped)
        assert len(none["disp"]) == 0
    ctx.close()
