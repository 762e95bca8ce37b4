"""Offset searches of several host threads at once, one over a wide image with a long disparity
range (more shared memory than a kernel has without asking), the others over narrow ones: every
call launches, and the wide search's counts are those of a call alone."""
import ctypes
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CALLS = 4000


def test_concurrent_searches_of_different_sizes():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2604_07980_gb300 import binding as B
    wide = torch.from_numpy(np.random.default_rng(61).integers(0, 256, (4, 2100), dtype=np.uint8)).cuda()
    narrow = wide[:, :128].contiguous()
    params = B.make_params(dict(win_w=3, win_h=3))
    ref = B.auto_rect(wide, wide, (0, 2, 2100, 3), 0, 599, 0, 0, 1, params=dict(win_w=3, win_h=3))[1].cpu()
    fn = B.lib().ctm_auto_rect
    failed, counts = {}, {}

    def work(name, im, nd):
        h, w = im.shape
        stream = torch.cuda.Stream()
        census = torch.empty((2, h, w), dtype=torch.int64, device="cuda")
        count = torch.empty(1, dtype=torch.int64, device="cuda")
        delta = torch.empty(1, dtype=torch.int32, device="cuda")
        torch.cuda.synchronize()
        p = [ctypes.c_void_p(t.data_ptr()) for t in (im, im, census, count, delta)]
        s = ctypes.c_void_p(stream.cuda_stream)
        failed[name] = 0
        for i in range(CALLS):
            failed[name] += fn(ctypes.byref(params), p[0], p[1], w, h, w, 0, 2, w, 3, 0, nd - 1, 0, 0, 1, 1, p[2],
                               p[3], p[4], s) != 0
            if i % 64 == 63:
                stream.synchronize()
        stream.synchronize()
        counts[name] = count.cpu()

    threads = [threading.Thread(target=work, args=a) for a in
               [("wide", wide, 600), ("narrow 0", narrow, 8), ("narrow 1", narrow, 16), ("narrow 2", narrow, 24)]]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert failed == {n: 0 for n in failed} and len(failed) == 4, failed
    assert torch.equal(counts["wide"], ref)
