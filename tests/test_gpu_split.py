"""GPU parity of the products whose contraction is split over a cluster (few tokens or small weights), at the sizes
where the split can go wrong: contractions that do not divide by the cluster or by a 64-deep stage, output widths
that leave part of a tile or of a CTA's columns empty, token counts on both sides of a copy's rows and of a tile.
Tolerances as for every linear (float32 accumulation, bf16 result)."""
import numpy as np
import pytest
import torch

import paper_2009_08065_b200 as bsp
import synth_inputs as si
from oracle import bsp_oracle as O
from gpu_util import DEV, assert_linear_close, bits_of, to_dev

pytestmark = pytest.mark.gpu


# clusters of 8, 4 and 2 on 64-wide tiles, 2 and 4 on 128-wide tiles, and shapes that stay whole
@pytest.mark.parametrize("tokens,n_out,k_in,act", [
    (1, 72, 1032, 0), (7, 768, 3072, 1), (127, 200, 1544, 0), (129, 760, 776, 1), (40, 2304, 768, 0),
    (600, 776, 3080, 0), (1003, 1024, 4096, 1), (300, 768, 3072, 0), (5, 304, 304, 0)])
@pytest.mark.parametrize("with_bias", [True, False])
def test_linear_with_split_contraction(tokens, n_out, k_in, act, with_bias):
    spec = si.LinearSpec(f"split{n_out}x{k_in}", n_out, k_in, bool(act), 2.0, 8)
    wp, _ = si.make_pruned_weight(81, spec)
    x = si.make_activations(81, spec.name, tokens, k_in)
    b = si.make_bias(81, spec)
    plan, xd, bd = to_dev(wp), to_dev(x), to_dev(b) if with_bias else None
    y = torch.full((tokens, n_out), 0x7FC0, dtype=torch.int16, device=DEV)
    bsp.bsp_linear_planned(plan, n_out, k_in, 8, xd, bd, act, y)
    bsp.bsp_linear_status()
    mask = O.mask_of(wp)
    bias = b if with_bias else np.zeros_like(b)
    rows = np.unique(np.linspace(0, tokens - 1, min(tokens, 160)).astype(int))
    y_ref = O.linear_masked_dense(x[rows], wp, mask, bias, act)
    assert_linear_close(bits_of(y)[rows], y_ref, O.row_scales(x[rows], wp, mask, bias), spec.name)
    # the same again with stale contents, and transposed, bit for bit
    y2 = torch.full_like(y, 0x1234)
    bsp.bsp_linear_planned_ex(plan, n_out, k_in, 8, xd, bd, act, y2, bsp.LINEAR_AUTO | bsp.LINEAR_PLAN_STABLE)
    assert torch.equal(y, y2)
    ldt = (tokens + 7) // 8 * 8
    yt = torch.full((n_out, ldt), 0x7FC0, dtype=torch.int16, device=DEV)
    bsp.bsp_linear_planned_ex(plan, n_out, k_in, 8, xd, bd, act, yt, bsp.LINEAR_AUTO | bsp.LINEAR_OUT_TRANSPOSED)
    bsp.bsp_linear_status()
    assert torch.equal(yt[:, :tokens], y.t())


# clusters of 8, 4 and 2, ragged tiles both ways, a contraction shorter than a stage; whole tiles 128, 192 and 256
# wide, one CTA with several of them; flags 8-byte aligned (mask in the epilogue) and not (mask kernel)
@pytest.mark.parametrize("tokens,n_out,k_in,block", [(200, 2312, 776, 8), (170, 3072, 1000, 16), (130, 4104, 1032, 8), (4000, 136, 264, 8), (2500, 392, 400, 8), (1300, 1200, 520, 16), (700, 264, 1032, 12), (40, 96, 72, 96)])
@pytest.mark.parametrize("aligned", [True, False])
def test_weight_gradient_with_split_contraction(tokens, n_out, k_in, block, aligned):
    dy = si.normal_bf16(82, f"dy{tokens}", (tokens, n_out), 1.0)
    x = si.normal_bf16(82, f"x{tokens}", (tokens, k_in), 1.0)
    keep = si.random_keep_sets(82, f"k{tokens}", n_out // block, k_in, k_in // 3)
    flags = torch.zeros(keep.size + 8, dtype=torch.uint8, device=DEV)
    flags = (flags[: keep.size] if aligned else flags[1: keep.size + 1]).view(keep.shape)
    flags.copy_(torch.from_numpy(keep.astype(np.uint8)))
    dw = torch.full((n_out, k_in), 0x7FC0, dtype=torch.int16, device=DEV)
    bsp.bsp_linear_backward_weight(to_dev(dy), to_dev(x), block, flags, dw)
    bsp.bsp_linear_status()
    mask = np.repeat(keep, block, axis=0)
    ref = O.linear_backward_weight(dy, x, mask)
    dyf, xf = O.bf16_to_f64(dy), O.bf16_to_f64(x)
    scales = np.linalg.norm(dyf, axis=0)[:, None] * np.linalg.norm(xf, axis=0)[None, :]
    assert_linear_close(bits_of(dw), ref, scales, "dW")
    assert (bits_of(dw)[~mask] == 0).all()
