"""BSP_LINEAR_PLAN_STABLE right behind the kernels that write the layouts: the flag is allowed on a linear whose layout
is complete before the call in front of it, here one linear earlier, while the writer overlaps that linear's start."""
import pytest
import torch

import paper_2009_08065_b200 as bsp
from gpu_util import DEV

pytestmark = pytest.mark.gpu


def packed(g, n_out, k_in, block):
    w = (torch.randn(n_out, k_in, generator=g, device=DEV) * 0.02).bfloat16()
    pk = bsp.PackedMatrix.allocate(n_out, k_in, block, bsp.ORIENT_C, DEV)
    bsp.bsp_prune_pack(w, pk, keep_per_block=k_in // 3)
    return pk


# 8 tokens: both linears split over clusters; 300: whole tiles; "pair": pairs of CTAs, with one tile each and with several.
# Layout A belongs to a small linear that is ready to start its weights at once, layout B is the larger one that its writer may
# still be storing.
@pytest.mark.parametrize("tokens,kernel", [(8, bsp.LINEAR_AUTO), (300, bsp.LINEAR_AUTO), (300, bsp.LINEAR_CTA_PAIR), (4096, bsp.LINEAR_CTA_PAIR)],
                         ids=["8", "300", "300-pair", "4096-pair"])
@pytest.mark.parametrize("writer", ["plan", "adam"])
def test_layouts_written_two_calls_before(tokens, kernel, writer):
    g = torch.Generator(device=DEV)
    g.manual_seed(tokens)
    shapes = [(256, 256), (3072, 3072)]                       # (n_out, k_in) of A and B
    block, versions = 16, 3
    pks = [[packed(g, n, k, block) for _ in range(versions)] for n, k in shapes]
    masters = [(torch.randn(*shapes[1], generator=g, device=DEV) * 0.02) for _ in range(versions)]
    grad = torch.zeros(shapes[1], device=DEV)
    moments = [torch.zeros(shapes[1], device=DEV) for _ in range(2)]
    plans = [torch.zeros(n * k * 2, dtype=torch.uint8, device=DEV) for n, k in shapes]
    xs = [torch.randn(tokens, k, generator=g, device=DEV).bfloat16() for _, k in shapes]

    def layouts(v):
        bsp.bsp_linear_plan(pks[0][v], plans[0])
        if writer == "plan":
            bsp.bsp_linear_plan(pks[1][v], plans[1])
        else:                                                 # the optimiser's bf16 copy is the layout
            bsp.bsp_masked_adam_step(masters[v], grad, moments[0], moments[1], None, 1, bsp.ORIENT_C, 0.0, 0.9, 0.999, 1e-8,
                                     0.0, 1, plans[1].view(torch.bfloat16).view(shapes[1]))

    def linear(i, y, algo):
        n, k = shapes[i]
        bsp.bsp_linear_planned_ex(plans[i], n, k, block, xs[i], None, bsp.ACT_NONE, y, algo)

    want = []
    for v in range(versions):
        layouts(v)
        torch.cuda.synchronize()
        want.append([torch.zeros(tokens, n, dtype=torch.bfloat16, device=DEV) for n, _ in shapes])
        for i in range(2):
            linear(i, want[v][i], kernel)
        torch.cuda.synchronize()
    assert not torch.equal(want[0][1], want[1][1])
    rounds = 60 if tokens < 4096 else 15                      # (outputs of 27 MB a round)
    got = [[torch.zeros_like(t) for t in want[0]] for _ in range(rounds)]
    for r in range(rounds):
        layouts(r % versions)
        linear(0, got[r][0], kernel | bsp.LINEAR_PLAN_STABLE)
        linear(1, got[r][1], kernel | bsp.LINEAR_PLAN_STABLE)
    bsp.bsp_linear_status()
    for r in range(rounds):
        for i in range(2):
            assert torch.equal(got[r][i], want[r % versions][i]), (r, i)
