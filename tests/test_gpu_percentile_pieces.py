"""GPU parity of batched percentiles whose row-blocks are small (short blocks or narrow matrices), which the sums take in
pieces of 32 chunks: heights that are no multiple of what a thread reads at once, matrices that end within a piece, a matrix
with too few groups for a histogram, rates of 1, weights beyond the size from which L1 is passed by.  Thresholds are exact."""
import numpy as np
import pytest
import torch

import paper_2009_08065_b200 as bsp
import synth_inputs as si
from oracle import bsp_oracle as O
from gpu_util import DEV, bits_of, to_dev

pytestmark = pytest.mark.gpu


MIN_BYTES, PAST_L1_BYTES, ITEM_BYTES, ROW_BYTES = 54 * 1024, 324 * 1024, 16 * 1024, 24 * 1024    # the first two per SM


def streamed_items(block, shapes):
    """Items that the streaming kernel would have: row-blocks, cut into equal column ranges where they exceed 24 KB."""
    most = ROW_BYTES // (2 * block) // 8 * 8
    total = 0
    for n, k in shapes:
        parts = -(-k // most)
        width = (-(-k // parts) + 7) // 8 * 8
        total += n // block * -(-k // width)
    return total


# (the last two are large enough for the rows to pass L1 by)
@pytest.mark.parametrize("block,shapes", [
    (1, [(2400, 1032), (3, 8), (1900, 1416), (97, 264)]),
    (3, [(3000, 528), (6, 8), (3201, 1032), (1500, 264)]),
    (8, [(4096, 256), (8, 8), (8200, 264), (4096, 400), (1024, 1032)]),
    (13, [(4160, 520), (13, 8), (5200, 264), (2600, 400), (26, 1032)]),
    (21, [(2100, 368), (4200, 272), (21, 8), (9450, 360)]),
    (8, [(8192, 1000)] * 4 + [(16, 72)]),
    (15, [(9000, 400), (15, 8)] + [(9000, 392)] * 7)])
def test_batched_percentile_in_pieces(block, shapes):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    total = sum(2 * n * k for n, k in shapes)
    large = shapes[0][0] >= 8192
    assert 1.05 * MIN_BYTES * sms <= total <= ITEM_BYTES * streamed_items(block, shapes)
    assert total >= 1.05 * PAST_L1_BYTES * sms if large else total <= PAST_L1_BYTES * sms / 1.05
    jobs, rates, weights = [], [], []
    for i, (n, k) in enumerate(shapes):
        w = si.normal_bf16(96, f"pp{block}.{i}", (n, k), 0.02)
        pk = bsp.PackedMatrix.allocate(n, k, block, bsp.ORIENT_C, DEV)
        t = torch.full((1,), float("nan"), device=DEV)
        jobs.append(bsp.LayerJob(to_dev(w), pk, 0.0, t))
        rates.append(1.0 if i == 3 else 1.7 + i)
        weights.append(w)
    bsp.bsp_percentile_threshold_batched(jobs, block, rates)
    bsp.bsp_linear_status()
    for job, rate, w in zip(jobs, rates, weights):
        want = O.percentile_threshold(w, block, "C", rate)
        assert np.float32(job.threshold_dev.item()) == np.float32(want)
