"""GPU parity of the re-packed values at the numbers of rows that a CTA takes (four or two, by the number of
row-blocks), with row-blocks that they do not divide, odd and even kept counts, and empty blocks.  Bits are moved, so the
result is exact."""
import numpy as np
import pytest
import torch

import paper_2009_08065_b200 as bsp
import synth_inputs as si
from gpu_util import DEV, bits_of, to_dev

pytestmark = pytest.mark.gpu


# at 3072 columns 1, 3, 30 and 75 row-blocks: two rows, of five rows two and two and one; 40 of 16 and 70 of 7 as well; 100 of 16,
# 200 of 7 and 300 of 4: four rows, as for narrower matrices
@pytest.mark.parametrize("blocks,block", [(1, 16), (3, 5), (30, 4), (40, 16), (75, 5), (70, 7), (100, 16), (200, 7), (300, 4)])
@pytest.mark.parametrize("cols,kept", [(8, 3), (264, 88), (3072, 771)])
def test_repack_by_rows_per_cta(blocks, block, cols, kept):
    rng = np.random.default_rng(blocks * 1000 + cols)
    keep = np.zeros((blocks, cols), bool)
    for b in range(blocks):
        n = 0 if blocks > 2 and b == blocks // 2 else kept - (b % 2)
        keep[b, rng.permutation(cols)[:n]] = True
    w = si.normal_bf16(94, f"rp{blocks}x{cols}", (blocks * block, cols), 0.02)
    new = si.normal_bf16(95, f"rp{blocks}x{cols}", (blocks * block, cols), 0.02)
    mask = np.repeat(keep, block, axis=0)
    pk = bsp.PackedMatrix.allocate(blocks * block, cols, block, bsp.ORIENT_C, DEV)
    bsp.bsp_prune_pack(to_dev(np.where(mask, w, 0).astype(w.dtype)), pk, 0.0)
    total = int(keep.sum()) * block
    pk.vals.fill_(0x7FC0)
    bsp.bsp_repack_values(to_dev(new), pk)
    want = np.concatenate([new[b * block:(b + 1) * block][:, keep[b]].reshape(-1) for b in range(blocks)])
    got = bits_of(pk.vals).reshape(-1)
    assert (got[:total] == want.view(got.dtype)).all()
    assert (got[total:] == 0x7FC0).all()
