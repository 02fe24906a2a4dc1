"""GPU parity of the gathering kernel's transposed output at the ends of its pieces: token counts within the first and the
second 64 of a 128-token tile and on their edges, each block height, row-blocks that do not divide by a run.  The last
shapes, with GELU and many row-blocks, leave as fragments (four epilogue groups).  Bit for bit the transpose of what the
kernel writes otherwise."""
import pytest
import torch

import paper_2009_08065_b200 as bsp
import synth_inputs as si
from gpu_util import DEV, to_dev

pytestmark = pytest.mark.gpu


SMALL = [(d, n, k, t, act) for d, n, k in ((32, 352, 264), (64, 960, 136), (128, 1408, 200))
         for t in (8, 56, 64, 72, 128, 136, 1000) for act in (0, 1)]
MANY = [(64, 2624, 72, 3720, 1), (64, 2624, 72, 3784, 1), (64, 2624, 136, 3776, 1), (128, 5248, 72, 3848, 1), (128, 5248, 72, 3904, 1)]


@pytest.mark.parametrize("d,n_out,k_in,tokens,act", SMALL + MANY)
def test_transposed_pieces(d, n_out, k_in, tokens, act):
    spec = si.LinearSpec(f"gt{d}", n_out, k_in, bool(act), 4.0, d)
    wp, _ = si.make_pruned_weight(93, spec)
    pk = bsp.PackedMatrix.allocate(n_out, k_in, d, bsp.ORIENT_C, DEV)
    bsp.bsp_prune_pack(to_dev(wp), pk, 0.0)
    gplan = torch.empty(bsp.bsp_linear_gather_plan_bytes(n_out, k_in, d), dtype=torch.uint8, device=DEV)
    bsp.bsp_linear_gather_plan(pk, gplan)
    xt = to_dev(si.make_activations(93, spec.name, tokens, k_in)).t().contiguous()
    b = to_dev(si.make_bias(93, spec))
    y = torch.full((tokens, n_out), 0x7FC0, dtype=torch.int16, device=DEV)
    yt = torch.full((n_out, tokens + 8), 0x7FC0, dtype=torch.int16, device=DEV)
    bsp.bsp_linear_gathered(gplan, n_out, k_in, d, xt, b, act, y)
    bsp.bsp_linear_gathered_ex(gplan, n_out, k_in, d, xt, b, act, yt[:, :tokens], True)
    bsp.bsp_linear_status()
    assert torch.equal(yt[:, :tokens], y.t())
    assert (yt[:, tokens:] == 0x7FC0).all()
