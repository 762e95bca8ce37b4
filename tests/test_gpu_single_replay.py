"""Single-frame calls on one context: from the second call on their launches replay as a graph
whose first and last nodes take the call's arguments.  Frames of other sizes and box counts,
other image, box and output buffers, an empty frame, another stream, a diagnostic call and a
changed tuning in between, and a call captured into a graph of the caller: every call's outputs
equal the oracle's."""
import numpy as np
import pytest

from oracle import oracle as orc
from paper_2604_07980_gb300 import workloads as wl
from tests.parity_util import compare_box_outputs, torch_frames

pytestmark = pytest.mark.gpu


def test_replayed_single_frame_calls_equal_oracle():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2604_07980_gb300 import binding as B
    sizes = [(640, 360, 20), (800, 450, 33), (321, 203, 7), (640, 360, 0), (800, 450, 12), (640, 360, 20)]
    ws = [wl.frame1080(seed=5200 + i, W=W, H=H, n_boxes=n, side_range=(12, 150)) for i, (W, H, n) in enumerate(sizes)]
    params = ws[0].params
    refs = [orc.match_frame(w.frames[0].left, w.frames[0].right, w.boxes, w.frames[0].f_px, w.frames[0].baseline_m,
                            orc.Params(**params)) for w in ws]
    dev = [(*torch_frames(w.frames)[0], torch.from_numpy(np.ascontiguousarray(w.boxes)).cuda()) for w in ws]
    ctx = B.Context(params, 1, 800, 450, 40)
    side = torch.cuda.Stream()

    def call(i, **kw):
        f = ws[i].frames[0]
        L, R, b = dev[i]
        return ctx.match_boxes(L, R, b, f.f_px, f.baseline_m, **kw)

    def check(got, i, where):
        torch.cuda.synchronize()
        compare_box_outputs({k: got[k].cpu().numpy() for k in ("disp", "depth", "flags")}, refs[i], where)
        assert ctx.stats()["error"] == 0

    for round_ in range(2):
        held = [call(i) for i in range(len(ws))]  # queued behind one another, each with buffers of its own
        for i, got in enumerate(held):
            check(got, i, f"round {round_} frame {i}")
    with torch.cuda.stream(side):
        got = call(1)
    check(got, 1, "another stream")
    check(call(4, debug=True), 4, "diagnostics")
    ctx.set_tuning(census_mode=2)
    check(call(0), 0, "changed tuning")
    check(call(5), 5, "changed tuning, replayed")
    # captured into the caller's own graph, replayed with other boxes in the same buffer
    L, R, b = dev[0]
    boxes = b.clone()
    f = ws[0].frames[0]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = ctx.match_boxes(L, R, boxes, f.f_px, f.baseline_m)
    graph.replay()
    check(out, 0, "captured by the caller")
    boxes.copy_(b.flip(0))
    graph.replay()
    ref = orc.match_frame(f.left, f.right, ws[0].boxes[::-1].copy(), f.f_px, f.baseline_m, orc.Params(**params))
    torch.cuda.synchronize()
    compare_box_outputs({k: out[k].cpu().numpy() for k in ("disp", "depth", "flags")}, ref, "captured, other boxes")
    ctx.close()


@pytest.mark.parametrize("mode", ["global", "thread_local", "relaxed"])
def test_replay_beside_a_capture(mode):
    """Calls on one stream while the same thread captures another stream: the replay's graph is
    built and launched, and the caller's capture stays valid, in every capture mode."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2604_07980_gb300 import binding as B
    w = wl.frame1080(seed=5300, W=640, H=360, n_boxes=9, side_range=(12, 150))
    f = w.frames[0]
    L, R = torch_frames(w.frames)[0]
    b = torch.from_numpy(np.ascontiguousarray(w.boxes)).cuda()
    ref = orc.match_frame(f.left, f.right, w.boxes, f.f_px, f.baseline_m, orc.Params(**w.params))
    n = len(w.boxes)
    outs = [(torch.empty(n, device="cuda"), torch.empty(n, device="cuda"),
             torch.empty(n, dtype=torch.uint8, device="cuda")) for _ in range(3)]
    x = torch.zeros(8, device="cuda")
    ctx = B.Context(w.params, 1, 640, 360, 16)
    side, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, capture_error_mode=mode):
        x.add_(1)
        for out in outs:
            ctx.match_boxes(L, R, b, f.f_px, f.baseline_m, out=out, stream=side)
    graph.replay()
    torch.cuda.synchronize()
    assert (x == 1).all()
    for i, out in enumerate(outs):
        got = {k: v.cpu().numpy() for k, v in zip(("disp", "depth", "flags"), out)}
        compare_box_outputs(got, ref, f"beside a {mode} capture, call {i}")
    ctx.close()
