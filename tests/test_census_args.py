"""The whole-image census reads its plane descriptors where the launch put them: the compiler
reports no stack for any window (indexing the argument by block made every thread copy it to
local memory)."""
import os
import re
import subprocess

import pytest

from paper_2604_07980_gb300 import build as B


def test_full_census_has_no_stack(tmp_path):
    try:
        nvcc = B.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    cmd = [nvcc, *B.ARCH, *B.NVCC_FLAGS, "-Xptxas", "-v", "-c", os.path.join(B.CSRC, "census.cu"), "-o",
           str(tmp_path / "census.o")]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    frames = re.findall(r"properties for \S*census_full_unit_kernel\S*\s+(\d+) bytes stack frame", r.stdout + r.stderr)
    assert frames == ["0"] * 3, frames
