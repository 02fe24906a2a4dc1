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


@pytest.mark.parametrize("block,shapes", [
    (1, [(2000, 1032), (3, 8), (1500, 1416), (97, 264)]),
    (3, [(3000, 528), (6, 8), (2001, 1032), (1500, 264)]),
    (8, [(4096, 256), (8, 8), (8200, 264), (4096, 400), (64, 1032)]),
    (21, [(2100, 368), (4200, 272), (21, 8), (6300, 360)]),
    (8, [(8192, 1000)] * 3 + [(16, 72)])])
def test_batched_percentile_in_pieces(block, shapes):
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
