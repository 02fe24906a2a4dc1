"""GPU parity of the column sums at every number of rows that a thread has in flight (4 in short blocks; 32, 16 or 8 by whether
the CTAs all run at once), in blocks that leave a remainder of every kind, whole and cut into column ranges.  Norms within
1e-5, thresholds and flags exact."""
import numpy as np
import pytest
import torch

import paper_2009_08065_b200 as bsp
import synth_inputs as si
from oracle import bsp_oracle as O
from gpu_util import DEV, packed_to_host, to_dev

pytestmark = pytest.mark.gpu


# (1400 and 900 row-blocks: more than run at once with 16 and with 32 rows in flight; 20 of wide rows: column ranges)
@pytest.mark.parametrize("block,blocks,cols", [
    (1, 40, 264), (2, 3000, 264), (3, 30, 1032), (7, 21, 72), (5, 20, 1544),
    (8, 24, 264), (8, 1400, 264), (9, 1400, 264), (13, 20, 264), (15, 1400, 264), (13, 20, 2056),
    (37, 12, 264), (37, 900, 264), (39, 1400, 264), (63, 20, 1544)])
def test_sums_by_rows_in_flight(block, blocks, cols):
    w = si.normal_bf16(97, f"tr{block}x{blocks}x{cols}", (block * blocks, cols), 0.02)
    w[:block, : cols // 2] = 0                                 # groups without any weight
    wd = to_dev(w)
    norms = torch.full((blocks, cols), -1.0, device=DEV)
    penalty = torch.full((1,), 3.0, dtype=torch.float64, device=DEV)
    bsp.bsp_group_norms(wd, block, bsp.ORIENT_C, 1e-3, bsp.PEN_L2, norms, torch.ones_like(norms), None, penalty)
    want = O.group_norms(w, block, "C")
    assert np.allclose(norms.cpu().numpy(), want, rtol=1e-5, atol=0)
    assert float(penalty.item()) == pytest.approx(float(want.sum()), rel=1e-5)
    pk = bsp.PackedMatrix.allocate(block * blocks, cols, block, bsp.ORIENT_C, DEV)
    t = torch.full((1,), float("nan"), device=DEV)
    bsp.bsp_percentile_threshold(wd, block, bsp.ORIENT_C, 2.5, t, pk.ws)
    threshold = O.percentile_threshold(w, block, "C", 2.5)
    assert np.float32(t.item()) == np.float32(threshold)
    bsp.bsp_prune_pack(wd, pk, 0.0, t)
    bsp.bsp_linear_status()
    assert np.array_equal(packed_to_host(pk)[3], O.keep_flags(w, block, "C", threshold))
