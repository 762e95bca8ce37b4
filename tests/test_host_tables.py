"""A host call's tables: their layout by size (plain C++, compiled and run here), and calls of
changing size, copied and mapped, on one context of a larger capacity, equal to the oracle."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import oracle as orc
from paper_2604_07980_gb300 import workloads as wl
from tests.parity_util import compare_box_outputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_layout(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    exe = tmp_path / "host_tables_check"
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", os.path.join(ROOT, "include"), "-I",
                    os.path.join(ROOT, "paper_2604_07980_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "host_tables_check.cpp"), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
    assert r.stdout.strip() == "OK"


@pytest.mark.gpu
def test_calls_of_changing_size_equal_oracle():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2604_07980_gb300 import binding as B
    W, H = 480, 272
    ws = [wl.frame1080(seed=5600 + i, W=W, H=H, n_boxes=4 + 3 * i, side_range=(12, 120)) for i in range(3)]
    f0 = ws[0].frames[0]
    refs = [orc.match_frame(w.frames[0].left, w.frames[0].right, w.boxes, f0.f_px, f0.baseline_m,
                            orc.Params(**ws[0].params)) for w in ws]
    host = [torch.from_numpy(np.stack([w.frames[0].left, w.frames[0].right])).pin_memory().numpy() for w in ws]
    ctx = B.Context(ws[0].params, 24, W, H, 600)
    for which in ([0], [0, 1, 2], [2], [2, 1], [1, 0, 2, 2, 1]):
        boxes = np.concatenate([ws[i].boxes for i in which])
        boxes[:, 4] = np.repeat(np.arange(len(which)), [len(ws[i].boxes) for i in which])
        for mapped in (True, False):
            got = ctx.match_batch_host([(host[i][0], host[i][1]) for i in which], boxes, f0.f_px, f0.baseline_m,
                                       mapped=mapped)
            ref = {k: np.concatenate([np.asarray(refs[i][k]) for i in which]) for k in ("disp", "depth", "flags")}
            compare_box_outputs(got, ref, f"frames {which}, mapped {mapped}")
    ctx.close()
