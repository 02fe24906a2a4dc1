"""A call that failed is reported once, by itself.  In a child process: the failing call ends a stream capture."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import torch
import paper_2009_08065_b200 as bsp
w = torch.ones(16, 16, dtype=torch.bfloat16, device="cuda")
mask = torch.zeros(16, 16, dtype=torch.uint8, device="cuda")
bsp.bsp_linear_status()
s = torch.cuda.Stream()
g = torch.cuda.CUDAGraph()
try:
    with torch.cuda.graph(g, stream=s):
        try:
            bsp.bsp_linear_status(s)              # reads a word back, which a capture does not allow
        except bsp.BspError as e:
            assert e.status == -4, e
        else:
            raise SystemExit("no error")
except Exception as e:
    print("capture ended:", type(e).__name__)
torch.cuda.synchronize()
for _ in range(2):
    bsp.bsp_dense_mask(w, mask)                   # a plain launch, checked through the runtime's last error
torch.cuda.synchronize()
assert mask.all()
print("done")
"""


def test_a_failed_call_leaves_no_error_behind():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout + r.stderr[-2000:]
