"""A NaN among the activations of one token reaches every output of that token and of no other one, with and without
GELU, on every route of the linear layer: a training run that diverged has to show."""
import pytest
import torch

import paper_2009_08065_b200 as bsp
from gpu_util import DEV

pytestmark = pytest.mark.gpu


def only_row_is_nan(y, row):
    nan = y.isnan()
    assert nan[row].all()
    nan[row] = False
    assert not nan.any()


def operands(tokens, n_out, k_in):
    g = torch.Generator(device=DEV)
    g.manual_seed(tokens + n_out)
    w = (torch.randn(n_out, k_in, generator=g, device=DEV) * 0.02).bfloat16()
    x = torch.randn(tokens, k_in, generator=g, device=DEV).bfloat16()
    x[5, 17] = float("nan")
    return w, x, (torch.randn(n_out, generator=g, device=DEV) * 0.02).bfloat16()


# 8 tokens: split over a cluster; 4096: whole tiles; both explicit kernels; the transposed output
@pytest.mark.parametrize("tokens", [8, 4096])
@pytest.mark.parametrize("algo", [bsp.LINEAR_AUTO, bsp.LINEAR_ONE_CTA, bsp.LINEAR_CTA_PAIR,
                                  bsp.LINEAR_AUTO | bsp.LINEAR_OUT_TRANSPOSED])
@pytest.mark.parametrize("act", [bsp.ACT_NONE, bsp.ACT_GELU])
def test_planned(tokens, algo, act):
    w, x, bias = operands(tokens, 768, 768)
    transposed = bool(algo & bsp.LINEAR_OUT_TRANSPOSED)
    y = torch.zeros((768, tokens) if transposed else (tokens, 768), dtype=torch.bfloat16, device=DEV)
    bsp.bsp_linear_planned_ex(w, 768, 768, 16, x, bias, act, y, algo)
    bsp.bsp_linear_status()
    only_row_is_nan(y.t().contiguous() if transposed else y, 5)


# blocks of 16 rows store from registers, taller ones through staging buffers; 8192 tokens x 4096 outputs take four
# epilogue groups with GELU
@pytest.mark.parametrize("block,tokens,n_out", [(16, 136, 64), (32, 136, 64), (128, 136, 256), (128, 8192, 4096)])
@pytest.mark.parametrize("transposed", [False, True])
def test_gathered(block, tokens, n_out, transposed):
    w, x, bias = operands(tokens, n_out, 128)
    pk = bsp.PackedMatrix.allocate(n_out, 128, block, bsp.ORIENT_C, DEV)
    bsp.bsp_prune_pack(w, pk, -1.0)                           # keeps every column
    gplan = torch.empty(bsp.bsp_linear_gather_plan_bytes(n_out, 128, block), dtype=torch.uint8, device=DEV)
    bsp.bsp_linear_gather_plan(pk, gplan)
    y = torch.zeros((n_out, tokens) if transposed else (tokens, n_out), dtype=torch.bfloat16, device=DEV)
    bsp.bsp_linear_gathered_ex(gplan, n_out, 128, block, x.t().contiguous(), bias, bsp.ACT_GELU, y, transposed)
    bsp.bsp_linear_status()
    only_row_is_nan(y.t().contiguous() if transposed else y, 5)


def test_packed_and_cuda_core():
    w, x, bias = operands(40, 768, 768)
    pk = bsp.PackedMatrix.allocate(768, 768, 16, bsp.ORIENT_C, DEV)
    bsp.bsp_prune_pack(w, pk, -1.0)
    ws = torch.empty(bsp.bsp_linear_plan_bytes(768, 768, 16), dtype=torch.uint8, device=DEV)
    for run in (lambda y: bsp.bsp_linear(pk, x, bias, bsp.ACT_GELU, y, ws),
                lambda y: bsp.bsp_linear_cuda_core(pk, x, bias, bsp.ACT_GELU, y)):
        y = torch.zeros((40, 768), dtype=torch.bfloat16, device=DEV)
        run(y)
        bsp.bsp_linear_status()
        only_row_is_nan(y, 5)


def test_chain():
    w, x, bias = operands(4096, 768, 768)
    y = torch.zeros((4096, 768), dtype=torch.bfloat16, device=DEV)
    ops = [bsp.ChainOp(plan=w, n_out=768, k_in=768, block=16, bias=bias, act=bsp.ACT_GELU, Y=y)]
    ws = torch.empty(bsp.bsp_linear_chain_ws_bytes(1, 4096), dtype=torch.uint8, device=DEV)
    bsp.bsp_linear_chain(ops, x, ws)
    bsp.bsp_linear_status()
    only_row_is_nan(y, 5)
