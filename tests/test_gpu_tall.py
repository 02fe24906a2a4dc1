"""The execution layouts of matrices so tall, or so wide, that their pieces do not fit one dimension of a grid."""
import numpy as np
import pytest
import torch

import paper_2009_08065_b200 as bsp
import synth_inputs as si
from oracle import bsp_oracle as O
from gpu_util import DEV, bits_of, to_dev, upload_packed

pytestmark = pytest.mark.gpu


def test_one_block_of_262148_rows():
    rows, cols = 262148, 8                                    # 65537 pieces of 4 rows
    w = si.normal_bf16(95, "tall", (rows, cols), 0.02)
    keep = np.array([[True, False, True, True, False, False, True, False]])
    pk = upload_packed(*O.pack(w, keep, rows, "C"), rows, cols, rows)
    plan = torch.full((bsp.bsp_linear_plan_bytes(rows, cols, rows),), 0x33, dtype=torch.uint8, device=DEV)
    bsp.bsp_linear_plan(pk, plan)
    assert np.array_equal(bits_of(plan.view(torch.int16)[: rows * cols]).reshape(rows, cols), si.zero_groups(w, keep, rows, "C"))


def test_transposed_layout_of_4194368_columns():
    rows, cols = 8, 4194368                                   # 65537 pieces of 64 columns
    w = si.normal_bf16(95, "wide", (rows, cols), 0.02)
    wd = to_dev(w)
    pk = bsp.PackedMatrix.allocate(rows, cols, 8, bsp.ORIENT_C, DEV)
    bsp.bsp_prune_pack(wd, pk, float(np.median(O.group_norms(w[:, :1024], 8, "C"))))
    plan_t = torch.full((bsp.bsp_linear_plan_bytes(rows, cols, 8),), 0x33, dtype=torch.uint8, device=DEV)
    bsp.bsp_linear_plan_t(pk, plan_t)
    want = torch.where(pk.keep.bool().view(1, cols), wd, torch.zeros_like(wd)).t()
    assert torch.equal(plan_t.view(torch.int16)[: rows * cols].view(cols, rows), want)


def test_layout_of_16777472_rows_in_strips():
    rows, cols = 16777472, 8                                  # 65537 pieces of 256 rows
    g = torch.Generator(device=DEV)
    g.manual_seed(95)
    w = torch.randint(1, 1000, (rows, cols), generator=g, device=DEV, dtype=torch.int16)
    kept = torch.arange(0, rows, 3, device=DEV, dtype=torch.int32)
    ptr = torch.tensor([0, kept.numel()], dtype=torch.int32, device=DEV)
    empty = torch.zeros(1, dtype=torch.uint8, device=DEV)
    pk = bsp.PackedMatrix(rows, cols, 8, bsp.ORIENT_R, ptr, kept, w[::3].contiguous(), empty, empty, empty)
    plan = torch.full((rows * cols * 2,), 0x33, dtype=torch.uint8, device=DEV)
    bsp.bsp_linear_plan(pk, plan)
    want = torch.zeros_like(w)
    want[::3] = w[::3]
    assert torch.equal(plan.view(torch.int16).view(rows, cols), want)


def test_percentile_of_2_to_the_32_groups():
    """Single weights as groups, more than 32-bit counts hold.  Row i repeats one value, the values grow with i, and
    every 1024th row starts a new one: the r-th smallest square follows from r."""
    n = 65536
    values = 0x3C00 + np.arange(n // 1024)                    # bf16 bit patterns, ascending
    rows = torch.from_numpy(np.repeat(values, 1024).astype(np.int16)).to(DEV)
    w = torch.empty(n, n, dtype=torch.int16, device=DEV)
    w.copy_(rows.view(n, 1).expand(n, n))
    ws = torch.empty(bsp.bsp_pack_bound(n, n, 1, bsp.ORIENT_C)[2], dtype=torch.uint8, device=DEV)
    t = torch.zeros(1, device=DEV)
    for rate in (1.5, 16.0):
        bsp.bsp_percentile_threshold(w, 1, bsp.ORIENT_C, rate, t, ws)
        r = int(float(n) * n * (1.0 - 1.0 / rate))
        v = np.uint32(int(values[(r - 1) // (1024 * n)]) << 16).view(np.float32)
        s = np.float32(v * v)
        want = np.sqrt(s)
        while np.float32(want * want) < s:
            want = np.nextafter(want, np.float32(np.inf))
        assert np.float32(t.item()) == want, rate
