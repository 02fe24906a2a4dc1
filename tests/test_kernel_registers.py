"""The column sums of short blocks must not pay for the long trips to memory of tall ones: what limits them is how many CTAs an
SM holds, so a form of each kernel has to exist that leaves it as many as before those trips.  Asked of the assembler, with the
build's own flags."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2009_08065_b200 import build as B

NVCC = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
pytestmark = pytest.mark.skipif(not os.path.exists(NVCC), reason="no nvcc here")


# 65536 registers: twelve CTAs of 96 threads with 56 of them; eight CTAs of 160 threads with 48
@pytest.mark.parametrize("source,kernel,most", [("bsp_fused.cu", "fused_stage1_kernel", 56), ("bsp_select.cu", "sums_c_kernel", 48)])
def test_short_blocks_keep_their_seats(source, kernel, most, tmp_path):
    flags = [f for f in B.NVCC_FLAGS if f != "-shared"]
    res = subprocess.run([NVCC, *flags, "-Xptxas", "-v", "-I", B.INCLUDE, "-I", B.CSRC, "-c", os.path.join(B.CSRC, source), "-o", str(tmp_path / "o.o")],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    used = [int(m.group(2)) for m in re.finditer(r"Compiling entry function '(\S+)'.*?Used (\d+) registers", res.stdout + res.stderr, re.S)
            if kernel in m.group(1)]
    assert used and min(used) <= most, used
