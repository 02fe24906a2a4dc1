"""GPU parity of the weight-side kernels at the sizes where their tiling can go wrong, against the oracle: the
percentile select (with and without its candidate list, list overflow, ragged ends), the keep-count select,
compaction in orientation R, the execution layouts, masking, value re-packing and the penalty gradient.
Everything but the gradient is bit-exact."""
import numpy as np
import pytest
import torch

import paper_2009_08065_b200 as bsp
import synth_inputs as si
from oracle import bsp_oracle as O
from gpu_util import DEV, bits_of, packed_to_host, to_dev, upload_packed

pytestmark = pytest.mark.gpu


def weights(name, rows, cols, ties=False):
    if ties:
        g = si.stream(71, si.tag_of(name))
        return si.f32_to_bf16_bits(g.integers(1, 3, size=(rows, cols)).astype(np.float32) * 0.5)
    return si.normal_bf16(71, name, (rows, cols), 0.02)


# groups: 18 / 20 thousand are selected straight from the sums, more through the list; 27567 leaves a ragged
# end; two-valued weights put half of the groups into one bin (list overflow); 2 million groups take two
# loads per thread
@pytest.mark.parametrize("rows,cols,block,orient,ties", [
    (96, 8, 8, 0, False), (576, 512, 16, 0, False), (640, 520, 16, 0, False), (1021, 27, 1, 0, False),
    (256, 256, 1, 0, True), (128, 128, 1, 0, True), (2048, 1024, 1, 0, False),
    (768, 768, 12, 1, False), (1000, 400, 8, 1, False), (333, 175, 5, 1, False), (300, 1200, 4, 1, True)])
def test_percentile_select(rows, cols, block, orient, ties):
    w = weights(f"sel{rows}x{cols}", rows, cols, ties)
    wd = to_dev(w)
    ws = torch.empty(bsp.bsp_pack_bound(rows, cols, block, orient)[2], dtype=torch.uint8, device=DEV)
    t = torch.zeros(1, dtype=torch.float32, device=DEV)
    for rate in (1.00001, 2.0, 7.9, 1e9):
        ws.fill_(0x5A)                                        # the workspace may hold anything
        bsp.bsp_percentile_threshold(wd, block, orient, rate, t, ws)
        assert np.float32(t.item()) == np.float32(O.percentile_threshold(w, block, "CR"[orient], rate)), rate


# a row per CTA and pieces numbered through: on both sides of 2048 rows and of 32 pieces a row; any geometry on both sides of
# a CTA per SM
@pytest.mark.parametrize("rows,cols,block,orient", [(2047, 248, 1, 0), (2048, 248, 2, 0), (2048, 256, 2, 0), (65536, 256, 256, 0),
                                                    (40, 2056, 8, 0), (148, 256, 4, 1), (149, 256, 4, 1), (300, 129, 3, 0)])
def test_mask_on_both_sides_of_its_rules(rows, cols, block, orient):
    w, o = weights(f"m{rows}x{cols}", rows, cols), "CR"[orient]
    keep = O.keep_flags(w, block, o, float(np.median(O.group_norms(w[:512] if orient == 0 else w, block, o))))
    wd = to_dev(w).clone()
    bsp.bsp_apply_mask(wd, block, orient, torch.from_numpy(keep.astype(np.uint8)).to(DEV))
    assert np.array_equal(bits_of(wd), si.zero_groups(w, keep, block, o))


def test_percentile_of_a_streamed_batch():
    """More items than the streaming sums need (six per SM) and more matrices than one launch takes: matrices with a
    histogram (16384 groups and more) among ones without, so that a CTA crosses from either kind to either; one cut into
    three column ranges of which the last is shorter; ties; rates of their own.  Bit for bit the single call's threshold."""
    block = 16
    shapes = []
    for i in range(104):
        shapes.append((1024, 264) if i % 3 == 0 else (160 + 16 * (i % 5), 8 * (1 + i % 31)))
    shapes[7], shapes[8], shapes[100] = (480, 2000), (1024, 776), (496, 2000)
    jobs, refs, rates = [], [], []
    for i, (rows, cols) in enumerate(shapes):
        w = weights(f"stream{i}", rows, cols, ties=i % 13 == 5)
        pk = bsp.PackedMatrix.allocate(rows, cols, block, bsp.ORIENT_C)
        pk.ws.fill_(0x5A)
        rates.append(1.0 + 0.37 * (i % 17))
        jobs.append(bsp.LayerJob(to_dev(w), pk, 0.0, torch.zeros(1, dtype=torch.float32, device=DEV)))
        refs.append(np.float32(O.percentile_threshold(w, block, "C", rates[-1])))
    items = sum(r // block * -(-c // 768) for r, c in shapes[:96])
    assert items >= 6 * torch.cuda.get_device_properties(0).multi_processor_count
    bsp.bsp_percentile_threshold_batched(jobs, block, rates)
    bsp.bsp_linear_status()
    assert [np.float32(j.threshold_dev.item()) for j in jobs] == refs


@pytest.mark.parametrize("rows,cols,block,orient,ties", [
    (16, 8192, 8, 0, False), (16, 8192, 8, 0, True), (24, 264, 12, 0, True), (10, 77, 5, 0, True),
    (2100, 24, 12, 1, True), (257, 16, 8, 1, False),
    (16, 192, 8, 0, True), (16, 200, 8, 0, False), (191, 24, 12, 1, True), (193, 16, 8, 1, False), (3, 24, 12, 1, True)])
def test_keep_count_select(rows, cols, block, orient, ties):
    w = weights(f"topk{rows}x{cols}", rows, cols, ties)
    o = "CR"[orient]
    groups = cols if orient == 0 else rows
    for keep_n in (1, groups // 3, groups - 1):
        pk = bsp.PackedMatrix.allocate(rows, cols, block, orient)
        bsp.bsp_prune_pack(to_dev(w), pk, keep_per_block=keep_n)
        keep_ref = O.keep_topk_per_block(w, block, o, keep_n)
        ref = O.pack(w, keep_ref, block, o)
        blk_ptr, idx, vals, keep, kept = packed_to_host(pk)
        assert np.array_equal(keep, keep_ref) and kept == block * int(keep_ref.sum())
        assert np.array_equal(blk_ptr, ref[0]) and np.array_equal(idx, ref[1]) and np.array_equal(vals, ref[2])


# rows above 1024 take several rounds of a CTA; 5000 strips have the counts scanned by a kernel of their own
@pytest.mark.parametrize("rows,cols,block", [(1025, 64, 16), (2500, 48, 12), (257, 35, 5), (8, 5000, 1)])
def test_pack_and_layout_of_row_pruned_strips(rows, cols, block):
    w = weights(f"r{rows}x{cols}", rows, cols)
    t = float(np.median(O.group_norms(w, block, "R")))
    keep_ref = O.keep_flags(w, block, "R", t)
    pk = bsp.PackedMatrix.allocate(rows, cols, block, bsp.ORIENT_R)
    bsp.bsp_prune_pack(to_dev(w), pk, t)
    ref = O.pack(w, keep_ref, block, "R")
    blk_ptr, idx, vals, keep, _ = packed_to_host(pk)
    assert np.array_equal(keep, keep_ref)
    assert np.array_equal(blk_ptr, ref[0]) and np.array_equal(idx, ref[1]) and np.array_equal(vals, ref[2])
    plan = torch.full(((rows * cols * 2 + 255) // 256 * 256,), 0x33, dtype=torch.uint8, device=DEV)
    bsp.bsp_linear_plan(pk, plan)
    assert np.array_equal(bits_of(plan.view(torch.int16)[: rows * cols]).reshape(rows, cols), O.prune(w, block, "R", t))


# strips of 1 to 7 columns on both sides of the scattering rule (more than eight CTAs per SM), 8 columns beyond it
@pytest.mark.parametrize("rows,cols,block", [(300, 1200, 1), (300, 580, 1), (1100, 1204, 4), (260, 4200, 7), (280, 9600, 8)])
def test_layout_of_narrow_strips(rows, cols, block):
    w = weights(f"n{rows}x{cols}", rows, cols)
    keep = si.random_keep_sets(72, f"n{rows}x{cols}", cols // block, rows, rows // 3).T.copy()
    keep[:, 1] = False                                        # an empty strip
    blk_ptr, idx, vals = O.pack(w, keep, block, "R")
    pk = upload_packed(blk_ptr, idx, vals, rows, cols, block, bsp.ORIENT_R)
    plan = torch.full(((rows * cols * 2 + 255) // 256 * 256,), 0x33, dtype=torch.uint8, device=DEV)
    bsp.bsp_linear_plan(pk, plan)
    assert np.array_equal(bits_of(plan.view(torch.int16)[: rows * cols]).reshape(rows, cols), si.zero_groups(w, keep, block, "R"))


# row-blocks on both sides of the rule for 1024 threads each (296), of columns that are no multiple of 8, by threshold and by
# keep count; segments on both sides of the 4096 up to which strips are packed by them; strips of 4096 groups and fewer
@pytest.mark.parametrize("rows,cols,block,orient", [(592, 1037, 2, 0), (594, 1037, 2, 0), (300, 2100, 1, 1), (300, 2048, 1, 1),
                                                    (4096, 300, 1, 1), (4090, 300, 1, 1)])
def test_pack_of_any_geometry(rows, cols, block, orient):
    w, o = weights(f"any{rows}x{cols}", rows, cols), "CR"[orient]
    t = float(np.median(O.group_norms(w, block, o)))
    groups = cols if orient == 0 else rows
    for keep_n in (-1, groups // 3):
        pk = bsp.PackedMatrix.allocate(rows, cols, block, orient)
        keep_ref = O.keep_flags(w, block, o, t) if keep_n < 0 else O.keep_topk_per_block(w, block, o, keep_n)
        bsp.bsp_prune_pack(to_dev(w), pk, t if keep_n < 0 else 0.0, keep_per_block=keep_n)
        ref = O.pack(w, keep_ref, block, o)
        blk_ptr, idx, vals, keep, kept = packed_to_host(pk)
        assert np.array_equal(keep, keep_ref) and kept == block * int(keep_ref.sum())
        assert np.array_equal(blk_ptr, ref[0]) and np.array_equal(idx, ref[1]) and np.array_equal(vals, ref[2])


# segments of 256 rows: a whole one, one row short, one row more, a single strip of many; 16400 strips are packed
# without segments
@pytest.mark.parametrize("rows,cols,block", [(256, 24, 12), (255, 16, 8), (257, 64, 64), (8192, 8, 8), (5, 16400, 1)])
def test_row_pruned_segments(rows, cols, block):
    w = weights(f"s{rows}x{cols}", rows, cols)
    t = float(np.median(O.group_norms(w, block, "R")))
    for keep_n in (-1, max(1, rows // 3), rows):
        pk = bsp.PackedMatrix.allocate(rows, cols, block, bsp.ORIENT_R)
        if keep_n < 0:
            keep_ref = O.keep_flags(w, block, "R", t)
            bsp.bsp_prune_pack(to_dev(w), pk, t)
        else:
            keep_ref = O.keep_topk_per_block(w, block, "R", keep_n)
            bsp.bsp_prune_pack(to_dev(w), pk, keep_per_block=keep_n)
        ref = O.pack(w, keep_ref, block, "R")
        blk_ptr, idx, vals, keep, kept = packed_to_host(pk)
        assert np.array_equal(keep, keep_ref) and kept == block * int(keep_ref.sum())
        assert np.array_equal(blk_ptr, ref[0]) and np.array_equal(idx, ref[1]) and np.array_equal(vals, ref[2])


@pytest.mark.parametrize("rows,cols,block", [(33, 72, 1), (63, 64, 3), (96, 136, 12), (144, 1024, 16), (128, 8, 64), (192, 200, 96), (200, 72, 100)])
def test_column_pruned_layouts_mask_and_repack(rows, cols, block):
    w = weights(f"c{rows}x{cols}", rows, cols)
    t = float(np.median(O.group_norms(w, block, "C")))
    keep = O.keep_flags(w, block, "C", t)
    keep[0, :] = False                                        # an empty row-block
    blk_ptr, idx, vals = O.pack(w, keep, block, "C")
    wp = si.zero_groups(w, keep, block, "C")
    pk = upload_packed(blk_ptr, idx, vals, rows, cols, block)
    plan_t = torch.full((bsp.bsp_linear_plan_bytes(rows, cols, block),), 0x33, dtype=torch.uint8, device=DEV)
    bsp.bsp_linear_plan_t(pk, plan_t)
    assert np.array_equal(bits_of(plan_t.view(torch.int16)[: rows * cols]).reshape(cols, rows), np.ascontiguousarray(wp.T))
    wd = to_dev(w).clone()
    bsp.bsp_apply_mask(wd, block, bsp.ORIENT_C, torch.from_numpy(keep.astype(np.uint8)).to(DEV))
    assert np.array_equal(bits_of(wd), wp)
    w2 = weights(f"again{rows}x{cols}", rows, cols)
    bsp.bsp_repack_values(to_dev(w2), pk)
    n = int(blk_ptr[-1]) * block
    assert np.array_equal(bits_of(pk.vals)[:n], O.repack_values(w2, blk_ptr, idx, block))


# rows that are no multiple of 8 and more than 1024 row-blocks are scattered; blocks of 16 rows, and 1024 row-blocks, not
@pytest.mark.parametrize("rows,cols,block", [(1025, 72, 1), (2056, 40, 2), (1024, 72, 1), (60, 136, 12), (102, 264, 3), (100, 72, 20)])
def test_transposed_layout_on_both_sides_of_the_scattering_rule(rows, cols, block):
    w = weights(f"t{rows}x{cols}", rows, cols)
    keep = si.random_keep_sets(73, f"t{rows}x{cols}", rows // block, cols, cols // 3)
    keep[1, :] = False
    pk = upload_packed(*O.pack(w, keep, block, "C"), rows, cols, block)
    plan_t = torch.full((bsp.bsp_linear_plan_bytes(rows, cols, block),), 0x33, dtype=torch.uint8, device=DEV)
    bsp.bsp_linear_plan_t(pk, plan_t)
    want = si.zero_groups(w, keep, block, "C").T
    assert np.array_equal(bits_of(plan_t.view(torch.int16)[: rows * cols]).reshape(cols, rows), np.ascontiguousarray(want))


# 3072 columns are staged, more are gathered from global memory, and so are single rows
@pytest.mark.parametrize("rows,cols,block,kept", [(8, 5120, 4, 1001), (8, 3072, 4, 1100), (8, 3080, 4, 1027), (6, 264, 1, 100), (6, 264, 2, 100)])
def test_repack_of_a_wide_matrix(rows, cols, block, kept):
    w = weights(f"wide{cols}", rows, cols)
    keep = si.random_keep_sets(5, "wide", rows // block, cols, kept)
    blk_ptr, idx, vals = O.pack(w, keep, block, "C")
    pk = upload_packed(blk_ptr, idx, np.zeros_like(vals), rows, cols, block)
    bsp.bsp_repack_values(to_dev(w), pk)
    assert np.array_equal(bits_of(pk.vals)[: vals.size], vals)


# blocks on both sides of the tiled kernel's row classes (8, 16, 32 rows), columns on both sides of its 256
@pytest.mark.parametrize("block,cols", [(1, 8), (8, 256), (9, 264), (16, 248), (17, 512), (32, 520), (33, 264)])
@pytest.mark.parametrize("pen", [bsp.PEN_L2, bsp.PEN_L2SQ])
def test_penalty_grad_tiles(block, cols, pen):
    rows = 3 * block
    w = weights(f"g{block}x{cols}", rows, cols)
    w[:block, :4] = 0                                         # all-zero groups
    gamma = O.gamma_update(O.group_norms(w, block, "C"), 1e-3).astype(np.float32)
    scale = 0.25
    ref = scale * O.penalty_grad(w, block, "C", gamma, pen == bsp.PEN_L2SQ)
    start = np.asarray(si.bf16_bits_to_f32(weights(f"start{block}", rows, cols)))
    for accumulate in (False, True):
        grad = torch.from_numpy(start.copy()).to(DEV)
        bsp.bsp_penalty_grad(to_dev(w), block, bsp.ORIENT_C, pen, torch.from_numpy(gamma).to(DEV), scale, grad, accumulate)
        want = ref + (start if accumulate else 0.0)
        # a norm of up to 33 squares, a division and two products: a few float32 roundings of the term and one of the sum
        err = np.abs(grad.cpu().numpy() - want)
        assert (err <= 1e-5 * np.abs(ref) + 2e-7 * np.abs(want) + 1e-30).all()
