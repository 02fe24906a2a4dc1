"""GPU parity of the CTA-pair products where their tiles can go wrong: rows that leave the second CTA of a pair without
any, outputs that end within a tile or a 32-column piece, contractions shorter than a stage or than the pipeline, several
tiles per pair, each tile width.  The linear form sums in the one-CTA kernel's order: equal bits.  The weight gradient is
held to the tolerance of every product (float32 accumulation, bf16 result)."""
import numpy as np
import pytest
import torch

import paper_2009_08065_b200 as bsp
import synth_inputs as si
from oracle import bsp_oracle as O
from gpu_util import DEV, assert_linear_close, bits_of, to_dev

pytestmark = pytest.mark.gpu


# tiles 256 x 128 (the first five), 256 x 192 (the next four) and 256 x 256
@pytest.mark.parametrize("tokens,n_out,k_in,act", [
    (1, 8, 8, 0), (129, 136, 72, 1), (257, 392, 200, 0), (300, 768, 776, 0), (8200, 1032, 72, 1), (4096, 768, 328, 0),
    (5000, 520, 72, 0), (1500, 2304, 264, 0), (4100, 2312, 776, 0), (5000, 2312, 200, 0), (6000, 4104, 136, 0)])
def test_pair_linear_matches_one_cta(tokens, n_out, k_in, act):
    x = to_dev(si.normal_bf16(91, f"px{tokens}", (tokens, k_in), 1.0))
    w = to_dev(si.normal_bf16(91, f"pw{n_out}", (n_out, k_in), 0.02))
    b = to_dev(si.normal_bf16(91, f"pb{n_out}", (n_out,), 0.02))
    plan = w.view(torch.uint8).reshape(-1)
    ys = []
    for algo in (bsp.LINEAR_ONE_CTA, bsp.LINEAR_CTA_PAIR, bsp.LINEAR_CTA_PAIR | bsp.LINEAR_PLAN_STABLE):
        y = torch.full((tokens, n_out), 0x7FC0, dtype=torch.int16, device=DEV)
        bsp.bsp_linear_planned_ex(plan, n_out, k_in, 8, x, b, act, y, algo)
        bsp.bsp_linear_status()
        ys.append(y)
    assert torch.equal(ys[0], ys[1]) and torch.equal(ys[0], ys[2])


# Each linear reads what the one before it is still storing, while its weights are fetched at once: up to six tiles per pair, and
# one tile behind them.
@pytest.mark.parametrize("tokens", [600, 6000])
def test_pair_chain_with_early_weights(tokens):
    widths = [776, 2304, 1032, 3072, 256, 768]
    x = to_dev(si.normal_bf16(93, f"cx{tokens}", (tokens, widths[0]), 1.0))
    plans = [to_dev(si.normal_bf16(93, f"cw{i}", (n, k), 0.02)).view(torch.uint8).reshape(-1) for i, (k, n) in enumerate(zip(widths, widths[1:]))]

    def chain(flags, rounds):
        out = []
        for _ in range(rounds):
            ys = [torch.full((tokens, n), 0x7FC0, dtype=torch.int16, device=DEV) for n in widths[1:]]
            src = x
            for i, y in enumerate(ys):
                bsp.bsp_linear_planned_ex(plans[i], widths[i + 1], widths[i], 8, src, None, i % 2, y, bsp.LINEAR_CTA_PAIR | flags)
                src = y
            out.append(ys)
        return out

    want = chain(0, 1)[0]
    got = chain(bsp.LINEAR_PLAN_STABLE, 8)
    bsp.bsp_linear_status()
    assert all(torch.equal(a, b) for ys in got for a, b in zip(ys, want))


# by pairs 256 x 128 (1000 x 2312 x 776 and the next four) and 256 x 256, and by one CTA with tiles 128 (65 x 1128 x 1816), 192
# (the first two, 1 x 1328 x 2168) and 256 wide (40 x 2104 x 4136); flags in the epilogue, by the mask kernel, none
@pytest.mark.parametrize("tokens,n_out,k_in,block", [
    (1, 2056, 1032, 8), (64, 2304, 1032, 16), (129, 1800, 1800, 3), (300, 3080, 1544, 8), (1000, 2312, 776, 8),
    (1, 2552, 2248, 8), (129, 1080, 568, 3), (65, 1448, 3520, 8), (40, 2456, 2720, 8),
    (700, 4000, 1000, 32), (600, 1000, 4000, 8), (64, 2200, 1640, 8), (65, 1128, 1816, 8), (1, 1328, 2168, 8), (40, 2104, 4136, 8)])
@pytest.mark.parametrize("flags", ["aligned", "unaligned", "none"])
def test_pair_weight_gradient(tokens, n_out, k_in, block, flags):
    dy = si.normal_bf16(92, f"dy{tokens}", (tokens, n_out), 1.0)
    x = si.normal_bf16(92, f"x{tokens}", (tokens, k_in), 1.0)
    keep = si.random_keep_sets(92, f"k{tokens}", n_out // block, k_in, k_in // 3) if flags != "none" else np.ones((n_out // block, k_in), bool)
    f = None
    if flags != "none":
        f = torch.zeros(keep.size + 8, dtype=torch.uint8, device=DEV)
        f = (f[: keep.size] if flags == "aligned" else f[1: keep.size + 1]).view(keep.shape)
        f.copy_(torch.from_numpy(keep.astype(np.uint8)))
    dw = torch.full((n_out, k_in), 0x7FC0, dtype=torch.int16, device=DEV)
    bsp.bsp_linear_backward_weight(to_dev(dy), to_dev(x), block, f, dw)
    bsp.bsp_linear_status()
    mask = np.repeat(keep, block, axis=0)
    rows = np.unique(np.linspace(0, n_out - 1, 400).astype(int))
    dyf, xf = O.bf16_to_f64(dy[:, rows]), O.bf16_to_f64(x)
    ref = np.where(mask[rows], dyf.T @ xf, 0.0)
    scales = np.linalg.norm(dyf, axis=0)[:, None] * np.linalg.norm(xf, axis=0)[None, :]
    got = bits_of(dw)
    assert_linear_close(got[rows], ref, scales, "dW")
    assert (got[~mask] == 0).all()
