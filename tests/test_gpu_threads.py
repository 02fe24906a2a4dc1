"""The first calls of a process, from several host threads at once, each on a stream of its own: what the library looks
up and sets up once (entry points, shared-memory limits, status words) must be complete before anyone uses it."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = """
import threading
import torch
import paper_2009_08065_b200 as bsp
n, k, d, tokens, count = 256, 256, 32, 136, 8
g = torch.Generator(device="cuda")
g.manual_seed(3)
w = (torch.randn(n, k, generator=g, device="cuda") * 0.02).bfloat16()
x = torch.randn(tokens, k, generator=g, device="cuda").bfloat16()
xt = x.t().contiguous()
pk = [bsp.PackedMatrix.allocate(n, k, d) for _ in range(count)]
plan = [torch.empty(bsp.bsp_linear_plan_bytes(n, k, d), dtype=torch.uint8, device="cuda") for _ in range(count)]
gplan = [torch.empty(bsp.bsp_linear_gather_plan_bytes(n, k, d), dtype=torch.uint8, device="cuda") for _ in range(count)]
ys = [[torch.zeros(tokens, n, dtype=torch.bfloat16, device="cuda") for _ in range(4)] for _ in range(count)]
dw = [torch.zeros(n, k, dtype=torch.bfloat16, device="cuda") for _ in range(count)]
t = [torch.zeros(1, device="cuda") for _ in range(count)]
streams = [torch.cuda.Stream() for _ in range(count)]
start, errors = threading.Barrier(count), []
torch.cuda.synchronize()

def work(i):
    try:
        s = streams[i]
        start.wait()
        bsp.bsp_linear_planned_ex(w, n, k, d, x, None, 1, ys[i][0], bsp.LINEAR_CTA_PAIR, stream=s)
        bsp.bsp_linear_planned_ex(w, n, k, d, x, None, 1, ys[i][1], bsp.LINEAR_ONE_CTA, stream=s)
        bsp.bsp_linear_backward_weight(x, x, d, None, dw[i], stream=s)
        bsp.bsp_percentile_threshold(w, d, bsp.ORIENT_C, 2.0, t[i], pk[i].ws, stream=s)
        bsp.bsp_prune_pack(w, pk[i], -1.0, stream=s)
        bsp.bsp_linear_plan(pk[i], plan[i], stream=s)
        bsp.bsp_linear_planned(plan[i], n, k, d, x, None, 1, ys[i][2], stream=s)
        bsp.bsp_linear_gather_plan(pk[i], gplan[i], stream=s)
        bsp.bsp_linear_gathered(gplan[i], n, k, d, xt, None, 1, ys[i][3], stream=s)
        s.synchronize()
    except Exception as e:
        errors.append(repr(e))

threads = [threading.Thread(target=work, args=(i,)) for i in range(count)]
[th.start() for th in threads]
[th.join() for th in threads]
assert not errors, errors
bsp.bsp_linear_status()
for i in range(1, count):
    assert torch.equal(dw[i], dw[0]) and torch.equal(t[i], t[0]) and t[0].item() > 0
    for a, b in zip(ys[i], ys[0]):
        assert torch.equal(a, b)
ref = torch.nn.functional.gelu(x.double() @ w.double().t())
for y in ys[0]:
    assert (y.double() - ref).norm() < 5e-3 * ref.norm()
print("done")
"""


def test_first_calls_from_several_threads():
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout + r.stderr[-2000:]
