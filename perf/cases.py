"""The work that is timed: what a program that prunes, retrains and serves a BERT-family encoder with this
library has it do, through the public calls, from one small linear up to whole stacks.

A case is a dict of plain values with a "kind":

  packed     one linear straight from the packed form (bsp_linear), nothing else kept around
  forward    the four linears of an encoder layer from their execution layouts, chained
  gathered   a feed-forward pair on the route that multiplies only the kept columns
  backward   activation and weight gradients of an encoder layer's four linears
  prune      norms, percentile or keep count, pruning, packing and execution layout of one matrix
  stack      the same for every matrix of an encoder stack, in batched calls
  reweight   one iteration of reweighted training (penalty, its gradient, Adam) on every matrix
  retrain    one iteration of masked retraining (Adam, bf16 copy, packed values) on every matrix

Weights are bf16 with a heavy tail and a standard deviation of 0.02, activations and gradients standard
normal and 1e-3 of it; kept sets are random where a case starts from a pruned matrix.
"""
from __future__ import annotations

import torch

import paper_2009_08065_b200 as bsp

EPS = 1e-3


def listed():
    return [
        # Trying one pruned linear out: batch 1, sequence 128, packed form in, as the package's smoke run does.
        {"name": "packed 768x768 T128", "kind": "packed", "rows": 768, "cols": 768, "block": 16, "rate": 2.0,
         "tokens": 128, "gelu": True},
        # Serving a single short query: a few tokens, so the number and the latency of the launches is all there is.
        {"name": "forward h768 T8", "kind": "forward", "hidden": 768, "block": 16, "rate": 3.0, "tokens": 8},
        # Serving a batch of sentences without padding: an odd number of tokens, a larger hidden size.
        {"name": "forward h1024 T1003", "kind": "forward", "hidden": 1024, "block": 32, "rate": 4.0, "tokens": 1003},
        # The benchmark's layer: batch 32 at sequence 128, three times compressed.
        {"name": "forward h768 T4096", "kind": "forward", "hidden": 768, "block": 16, "rate": 3.0, "tokens": 4096},
        # Scoring a corpus offline: the largest batch of the compression sweep.
        {"name": "forward h1024 T32768", "kind": "forward", "hidden": 1024, "block": 16, "rate": 3.0, "tokens": 32768},
        # The same with tall blocks and high compression, where the pruned work is skipped.
        {"name": "gathered h1024 T8192", "kind": "gathered", "hidden": 1024, "block": 128, "rate": 8.0, "tokens": 8192},
        # The backward half of a retraining step at the usual batch.
        {"name": "backward h768 T4096", "kind": "backward", "hidden": 768, "block": 16, "rate": 3.0, "tokens": 4096},
        # Pruning one matrix to a compression rate: the README's example.
        {"name": "prune C 3072x768", "kind": "prune", "rows": 3072, "cols": 768, "block": 16, "rate": 3.0,
         "orient": "C", "mode": "percentile"},
        # The row variant with one of the paper's block widths.
        {"name": "prune R 768x768", "kind": "prune", "rows": 768, "cols": 768, "block": 12, "rate": 2.0,
         "orient": "R", "mode": "percentile"},
        # A pruning milestone on the whole encoder: 12 layers of six matrices.
        {"name": "stack 12 layers h768", "kind": "stack", "layers": 12, "hidden": 768, "block": 16, "rate": 5.0},
        # An iteration of reweighted training on one large layer.
        {"name": "reweight 1 layer h1024", "kind": "reweight", "layers": 1, "hidden": 1024, "block": 16},
        # An iteration of retraining under the mask on the whole encoder.
        {"name": "retrain 12 layers h768", "kind": "retrain", "layers": 12, "hidden": 768, "block": 16, "rate": 3.0},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(lo * (hi / lo) ** rng.random()))))


def _block_of(rng, size, choices):
    return rng.choice([b for b in choices if size % b == 0])


def draw(rng):
    kind = rng.choice(["packed", "forward", "forward", "forward", "gathered", "backward", "prune", "prune", "stack",
                       "reweight", "retrain"])
    hidden = 16 * rng.randint(16, 64)                     # 256 ... 1024
    rate = round(rng.uniform(1.5, 8.0), 2)
    if kind == "packed":
        rows, cols = 16 * rng.randint(16, 192), 8 * rng.randint(32, 384)
        return {"kind": kind, "rows": rows, "cols": cols, "block": _block_of(rng, rows, (4, 8, 16, 32, 64, 96)),
                "rate": rate, "tokens": _log_int(rng, 1, 4096), "gelu": rng.random() < 0.5}
    if kind == "forward":
        return {"kind": kind, "hidden": hidden, "block": _block_of(rng, hidden, (3, 8, 16, 32, 64, 96)), "rate": rate,
                "tokens": _log_int(rng, 1, 32768)}
    if kind == "gathered":
        hidden = 128 * rng.randint(4, 8)
        block = rng.choice((64, 128))
        return {"kind": kind, "hidden": hidden, "block": block, "rate": round(rng.uniform(4.0 if block == 128 else 7.0, 10.0), 2),
                "tokens": 8 * _log_int(rng, 16, 2048)}
    if kind == "backward":
        return {"kind": kind, "hidden": hidden, "block": _block_of(rng, hidden, (8, 16, 32, 64)), "rate": rate,
                "tokens": _log_int(rng, 128, 8192)}
    if kind == "prune":
        rows, cols = 16 * rng.randint(16, 192), 16 * rng.randint(16, 64)
        if rng.random() < 0.5:
            rows, cols = cols, rows
        orient = rng.choice("CR")
        return {"kind": kind, "rows": rows, "cols": cols, "rate": rate, "orient": orient,
                "block": _block_of(rng, rows if orient == "C" else cols, (8, 12, 16, 32, 64, 96)),
                "mode": rng.choice(("percentile", "percentile", "keep_count"))}
    if kind == "stack":
        return {"kind": kind, "layers": rng.randint(1, 12), "hidden": 16 * rng.randint(16, 48), "rate": rate,
                "block": rng.choice((8, 16, 16))}
    hidden = 16 * rng.randint(16, 48)
    if kind == "reweight":
        return {"kind": kind, "layers": rng.randint(1, 8), "hidden": hidden, "block": rng.choice((8, 16))}
    return {"kind": kind, "layers": rng.randint(1, 12), "hidden": hidden, "block": rng.choice((8, 16)), "rate": rate}


# ----------------------------------------------------------------------------------------------------------
# shapes
# ----------------------------------------------------------------------------------------------------------
def _layer_shapes(hidden):
    """(n_out, k_in) of a layer's linears: fused QKV, attention output, FFN up, FFN down."""
    return [(3 * hidden, hidden), (hidden, hidden), (4 * hidden, hidden), (hidden, 4 * hidden)]


def _stack_shapes(hidden, layers):
    """Six matrices per layer: Q, K, V, attention output, FFN up, FFN down."""
    return ([(hidden, hidden)] * 4 + [(4 * hidden, hidden), (hidden, 4 * hidden)]) * layers


def _kept(cols, rate):
    return max(1, int(round(cols / rate)))


# ----------------------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(g, shape, std=1.0):
    return (torch.randn(shape, generator=g, device="cuda") * std).bfloat16()


def _weights(g, shape):
    """Student-t with three degrees of freedom scaled to a standard deviation of 0.02."""
    z = torch.randn(shape, generator=g, device="cuda")
    chi2 = torch.zeros(shape, device="cuda")
    for _ in range(3):
        chi2 += torch.randn(shape, generator=g, device="cuda") ** 2
    return (z * (3.0 / chi2).sqrt_() * (0.02 / 3.0 ** 0.5)).bfloat16()


def _pruned(g, rows, cols, block, rate):
    """A matrix in which every row-block keeps the same number of randomly chosen columns, packed."""
    W = _weights(g, (rows, cols))
    scores = torch.rand((rows // block, cols), generator=g, device="cuda")
    kept = scores.topk(_kept(cols, rate), dim=1).indices
    mask = torch.zeros_like(scores, dtype=torch.bool).scatter_(1, kept, True)
    W = torch.where(mask.repeat_interleave(block, dim=0), W, torch.zeros((), dtype=W.dtype, device="cuda"))
    pk = bsp.PackedMatrix.allocate(rows, cols, block, bsp.ORIENT_C)
    bsp.bsp_prune_pack(W, pk, 0.0)
    return W, pk


def _plan(pk):
    plan = torch.empty((pk.rows * pk.cols * 2 + 255) // 256 * 256, dtype=torch.uint8, device="cuda")
    bsp.bsp_linear_plan(pk, plan)
    return plan


def _flat_views(shapes, dtype, fill=None):
    """One buffer and a view of it per shape, each view starting on a 256-byte boundary."""
    step = 256 // torch.empty((), dtype=dtype).element_size()
    starts, total = [], 0
    for s in shapes:
        starts.append(total)
        n = 1
        for v in s:
            n *= v
        total += (n + step - 1) // step * step
    flat = torch.zeros(total, dtype=dtype, device="cuda")
    views = []
    for s, at in zip(shapes, starts):
        n = 1
        for v in s:
            n *= v
        views.append(flat[at:at + n].view(s))
    return flat, views


def prepare(case, seed):
    return _PREPARE[case["kind"]](case, _gen(seed))


def run(state):
    return state["run"](state)


# ---------------------------------------------------------------------------------------------- packed
def _prepare_packed(c, g):
    _, pk = _pruned(g, c["rows"], c["cols"], c["block"], c["rate"])
    return {"run": _run_packed, "pk": pk, "X": _normal(g, (c["tokens"], c["cols"])), "bias": _normal(g, (c["rows"],), 0.02),
            "act": bsp.ACT_GELU if c["gelu"] else bsp.ACT_NONE,
            "Y": torch.empty((c["tokens"], c["rows"]), dtype=torch.bfloat16, device="cuda"),
            "ws": torch.empty(bsp.bsp_linear_plan_bytes(c["rows"], c["cols"], c["block"]), dtype=torch.uint8, device="cuda")}


def _run_packed(s):
    bsp.bsp_linear(s["pk"], s["X"], s["bias"], s["act"], s["Y"], s["ws"])
    return s["Y"]


# --------------------------------------------------------------------------------------------- forward
def _prepare_forward(c, g):
    h, T = c["hidden"], c["tokens"]
    shapes = _layer_shapes(h)
    X = _normal(g, (T, h))
    Y = [torch.empty((T, n), dtype=torch.bfloat16, device="cuda") for n, _ in shapes]
    # without attention in between, the attention-output linear reads the V third of QKV's output
    sources = [X, Y[0][:, 2 * h:], Y[1], Y[2]]
    acts = [bsp.ACT_NONE, bsp.ACT_NONE, bsp.ACT_GELU, bsp.ACT_NONE]
    linears = []
    for (n, k), src, act, y in zip(shapes, sources, acts, Y):
        plan = _plan(_pruned(g, n, k, c["block"], c["rate"])[1])
        linears.append((plan, n, k, src, _normal(g, (n,), 0.02), act, y))
    return {"run": _run_forward, "linears": linears, "block": c["block"], "Y": Y}


def _run_forward(s):
    for plan, n, k, src, bias, act, y in s["linears"]:
        bsp.bsp_linear_planned_ex(plan, n, k, s["block"], src, bias, act, y, bsp.LINEAR_AUTO | bsp.LINEAR_PLAN_STABLE)
    return s["Y"]


# -------------------------------------------------------------------------------------------- gathered
def _prepare_gathered(c, g):
    h, T, d = c["hidden"], c["tokens"], c["block"]
    gplans, biases = [], []
    for n, k in _layer_shapes(h)[2:]:
        _, pk = _pruned(g, n, k, d, c["rate"])
        gplan = torch.empty(bsp.bsp_linear_gather_plan_bytes(n, k, d), dtype=torch.uint8, device="cuda")
        bsp.bsp_linear_gather_plan(pk, gplan)
        gplans.append(gplan)
        biases.append(_normal(g, (n,), 0.02))
    X = _normal(g, (T, h))
    XT = torch.empty((h, T), dtype=torch.bfloat16, device="cuda")
    midT = torch.empty((4 * h, T), dtype=torch.bfloat16, device="cuda")
    Y = torch.empty((T, h), dtype=torch.bfloat16, device="cuda")
    kept = [n * _kept(k, c["rate"]) for n, k in _layer_shapes(h)[2:]]
    up = bsp.make_linear_call(4 * h, h, d, T, gplan=gplans[0], kept_weights=kept[0], XT=XT, bias=biases[0],
                              act=bsp.ACT_GELU, YT=midT)
    down = bsp.make_linear_call(h, 4 * h, d, T, gplan=gplans[1], kept_weights=kept[1], XT=midT, bias=biases[1], Y=Y)
    return {"run": _run_gathered, "X": X, "XT": XT, "midT": midT, "Y": Y, "up": up, "down": down,
            "keep": (gplans, biases)}


def _run_gathered(s):
    bsp.bsp_transpose(s["X"], s["XT"])
    bsp.bsp_linear_run(s["up"])
    bsp.bsp_linear_run(s["down"])
    return [s["midT"], s["Y"]]


# -------------------------------------------------------------------------------------------- backward
def _prepare_backward(c, g):
    T, d = c["tokens"], c["block"]
    linears, out = [], []
    for n, k in _layer_shapes(c["hidden"]):
        _, pk = _pruned(g, n, k, d, c["rate"])
        plan_t = torch.empty(bsp.bsp_linear_plan_bytes(n, k, d), dtype=torch.uint8, device="cuda")
        dX = torch.empty((T, k), dtype=torch.bfloat16, device="cuda")
        dW = torch.empty((n, k), dtype=torch.bfloat16, device="cuda")
        linears.append((pk, plan_t, _normal(g, (T, n), 1e-3), _normal(g, (T, k)), dX, dW))
        out += [dX, dW]
    return {"run": _run_backward, "linears": linears, "out": out}


def _run_backward(s):
    # the optimiser has just changed the packed values, so the transposed layout is made anew each step
    for pk, plan_t, dY, X, dX, dW in reversed(s["linears"]):
        bsp.bsp_linear_plan_t(pk, plan_t)
        bsp.bsp_linear_planned(plan_t, pk.cols, pk.rows, 1, dY, None, bsp.ACT_NONE, dX)
        bsp.bsp_linear_backward_weight(dY, X, pk.block, pk.keep, dW)
    return s["out"]


# ----------------------------------------------------------------------------------------------- prune
def _prepare_prune(c, g):
    rows, cols, d = c["rows"], c["cols"], c["block"]
    orient = bsp.ORIENT_C if c["orient"] == "C" else bsp.ORIENT_R
    pk = bsp.PackedMatrix.allocate(rows, cols, d, orient)
    pk.idx.zero_()
    pk.vals.zero_()
    shape = tuple(pk.keep.shape)
    groups = cols if c["orient"] == "C" else rows
    return {"run": _run_prune, "W": _weights(g, (rows, cols)), "pk": pk, "rate": c["rate"],
            "keep_count": _kept(groups, c["rate"]) if c["mode"] == "keep_count" else -1,
            "norms": torch.empty(shape, dtype=torch.float32, device="cuda"),
            "gamma": torch.empty(shape, dtype=torch.float32, device="cuda"),
            "penalty": torch.zeros(1, dtype=torch.float64, device="cuda"),
            "t": torch.zeros(1, dtype=torch.float32, device="cuda"),
            "plan": torch.zeros((rows * cols * 2 + 255) // 256 * 256, dtype=torch.uint8, device="cuda")}


def _run_prune(s):
    W, pk = s["W"], s["pk"]
    bsp.bsp_group_norms(W, pk.block, pk.orient, EPS, bsp.PEN_L2, s["norms"], None, s["gamma"], s["penalty"])
    if s["keep_count"] < 0:
        bsp.bsp_percentile_threshold(W, pk.block, pk.orient, s["rate"], s["t"], pk.ws)
        bsp.bsp_prune_pack(W, pk, 0.0, s["t"])
    else:
        bsp.bsp_prune_pack(W, pk, keep_per_block=s["keep_count"])
    bsp.bsp_linear_plan(pk, s["plan"])
    return [s["norms"], s["gamma"], s["penalty"], s["t"], pk.keep, pk.blk_ptr, pk.idx, pk.vals, pk.kept_weights, s["plan"]]


# ----------------------------------------------------------------------------------------------- stack
def _prepare_stack(c, g):
    d = c["block"]
    shapes = _stack_shapes(c["hidden"], c["layers"])
    per_group = [(n // d, k) for n, k in shapes]
    flat = {}
    flat["W"], W = _flat_views(shapes, torch.bfloat16)
    flat["norms"], norms = _flat_views(per_group, torch.float32)
    flat["gamma"], gamma = _flat_views(per_group, torch.float32)
    flat["penalty"], penalty = _flat_views([(1,)] * len(shapes), torch.float64)
    flat["t"], t = _flat_views([(1,)] * len(shapes), torch.float32)
    flat["keep"], keep = _flat_views(per_group, torch.uint8)
    flat["blk_ptr"], blk_ptr = _flat_views([(n // d + 1,) for n, _ in shapes], torch.int32)
    flat["idx"], idx = _flat_views([(bsp.bsp_pack_bound(n, k, d)[0],) for n, k in shapes], torch.int32)
    flat["vals"], vals = _flat_views([(n * k,) for n, k in shapes], torch.int16)
    flat["kept"], kept = _flat_views([(1,)] * len(shapes), torch.int64)
    flat["plan"], plan = _flat_views(shapes, torch.bfloat16)
    flat["ws"], ws = _flat_views([(bsp.bsp_pack_bound(n, k, d)[2],) for n, k in shapes], torch.uint8)
    jobs = []
    for i, (n, k) in enumerate(shapes):
        W[i].copy_(_weights(g, (n, k)))
        pk = bsp.PackedMatrix(n, k, d, bsp.ORIENT_C, blk_ptr[i], idx[i], vals[i], keep[i], kept[i], ws[i])
        jobs.append(bsp.LayerJob(W[i], pk, 0.0, t[i], norms[i], None, gamma[i], penalty[i], plan[i]))
    # the rate of every matrix within a fifth of the stack's
    rates = [c["rate"] * (0.8 + 0.4 * ((7 * i) % 11) / 10.0) for i in range(len(shapes))]
    return {"run": _run_stack, "jobs": bsp.make_job_array(jobs), "rates": [max(1.0, r) for r in rates], "block": d, "flat": flat}


def _run_stack(s):
    bsp.bsp_percentile_threshold_batched(s["jobs"], s["block"], s["rates"])
    bsp.bsp_prepare_batched(s["jobs"], s["block"], EPS, bsp.PEN_L2)
    f = s["flat"]
    return [f[k] for k in ("norms", "gamma", "penalty", "t", "keep", "blk_ptr", "idx", "vals", "kept", "plan")]


# ------------------------------------------------------------------------------------ reweight, retrain
def _optimiser_state(c, g):
    shapes = _layer_shapes(c["hidden"]) * c["layers"]
    flat, views = {}, {}
    for name in ("W", "G", "m", "v"):
        flat[name], views[name] = _flat_views(shapes, torch.float32)
    flat["Wb"], views["Wb"] = _flat_views(shapes, torch.bfloat16)
    for i, s in enumerate(shapes):
        views["Wb"][i].copy_(_weights(g, s))
        views["G"][i].copy_(torch.randn(s, generator=g, device="cuda") * 1e-3)
        views["m"][i].copy_(torch.randn(s, generator=g, device="cuda") * 1e-3)
        views["v"][i].copy_(torch.rand(s, generator=g, device="cuda") * 1e-6)
    flat["W"].copy_(flat["Wb"])
    return shapes, flat, views


def _prepare_reweight(c, g):
    d = c["block"]
    shapes, flat, v = _optimiser_state(c, g)
    flat["gamma"], gamma = _flat_views([(n // d, k) for n, k in shapes], torch.float32)
    flat["penalty"], penalty = _flat_views([(1,)] * len(shapes), torch.float64)
    for i in range(len(shapes)):
        bsp.bsp_group_norms(v["Wb"][i], d, bsp.ORIENT_C, EPS, bsp.PEN_L2, gamma_out=gamma[i])
    mats = [(v["W"][i], v["Wb"][i], v["G"][i], v["m"][i], v["v"][i], gamma[i], penalty[i]) for i in range(len(shapes))]
    return {"run": _run_reweight, "mats": mats, "block": d, "flat": flat, "step": 10}


def _run_reweight(s):
    d, flat = s["block"], s["flat"]
    s["step"] += 1
    for W, Wb, G, m, v, gamma, penalty in s["mats"]:
        bsp.bsp_group_norms(Wb, d, bsp.ORIENT_C, EPS, bsp.PEN_L2, gamma_in=gamma, penalty=penalty)
        bsp.bsp_penalty_grad(Wb, d, bsp.ORIENT_C, bsp.PEN_L2, gamma, 1e-5, G, accumulate=True)
        bsp.bsp_masked_adam_step(W, G, m, v, None, d, bsp.ORIENT_C, 3e-5, 0.9, 0.999, 1e-8, 0.0, s["step"], Wb)
    return [flat[k] for k in ("W", "Wb", "G", "m", "v", "penalty")]


def _prepare_retrain(c, g):
    d = c["block"]
    shapes, flat, v = _optimiser_state(c, g)
    flat["vals"], vals = _flat_views([(n * k,) for n, k in shapes], torch.int16)
    mats = []
    for i, (n, k) in enumerate(shapes):
        Wp, pk = _pruned(g, n, k, d, c["rate"])
        v["Wb"][i].copy_(Wp)
        v["W"][i].copy_(Wp)
        pk.vals = vals[i]
        mats.append((v["W"][i], v["Wb"][i], v["G"][i], v["m"][i], v["v"][i], pk))
    return {"run": _run_retrain, "mats": mats, "block": d, "flat": flat, "step": 10}


def _run_retrain(s):
    d, flat = s["block"], s["flat"]
    s["step"] += 1
    for W, Wb, G, m, v, pk in s["mats"]:
        bsp.bsp_masked_adam_step(W, G, m, v, pk.keep, d, bsp.ORIENT_C, 3e-5, 0.9, 0.999, 1e-8, 0.0, s["step"], Wb)
        bsp.bsp_repack_values(Wb, pk)
    return [flat[k] for k in ("W", "Wb", "m", "v", "vals")]


_PREPARE = {"packed": _prepare_packed, "forward": _prepare_forward, "gathered": _prepare_gathered,
            "backward": _prepare_backward, "prune": _prepare_prune, "stack": _prepare_stack,
            "reweight": _prepare_reweight, "retrain": _prepare_retrain}


# ----------------------------------------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------------------------------------
def _linear_work(n, k, block, rate, tokens):
    """Activations in and out once, kept values, one index per kept group, bias; the kept multiply-adds."""
    kept = n * _kept(k, rate)
    return 2 * tokens * (n + k) + 2 * kept + 4 * (kept // block) + 2 * n, 2 * tokens * kept


def _prune_work(n, k, block, rate):
    """Weights in; norm, gamma and flag per group, values and indices of the kept groups and the layout out."""
    groups = n * k // block
    kept = n * k / rate
    return 2 * n * k + 9 * groups + 2 * kept + 4 * kept / block + 2 * n * k, 4 * n * k


def work(case):
    c, kind = case, case["kind"]
    total_bytes = total_flops = 0.0

    def add(bytes_flops):
        nonlocal total_bytes, total_flops
        total_bytes += bytes_flops[0]
        total_flops += bytes_flops[1]

    if kind == "packed":
        add(_linear_work(c["rows"], c["cols"], c["block"], c["rate"], c["tokens"]))
    elif kind == "forward":
        for n, k in _layer_shapes(c["hidden"]):
            add(_linear_work(n, k, c["block"], c["rate"], c["tokens"]))
    elif kind == "gathered":
        for n, k in _layer_shapes(c["hidden"])[2:]:
            add(_linear_work(n, k, c["block"], c["rate"], c["tokens"]))
    elif kind == "backward":
        T = c["tokens"]
        for n, k in _layer_shapes(c["hidden"]):
            kept = n * _kept(k, c["rate"])
            # dY and X in once, kept values and indices, flags; dX and dW out
            add((2 * T * n + 2 * T * k + 2 * kept + 4 * kept // c["block"] + n * k // c["block"] + 2 * T * k + 2 * n * k, 4 * T * kept))
    elif kind == "prune":
        add(_prune_work(c["rows"], c["cols"], c["block"], c["rate"]))
    elif kind == "stack":
        for n, k in _stack_shapes(c["hidden"], c["layers"]):
            add(_prune_work(n, k, c["block"], c["rate"]))
    else:
        for n, k in _layer_shapes(c["hidden"]) * c["layers"]:
            if kind == "reweight":
                # float32 weight, gradient and moments in and out, bf16 weights in and out, one gamma per group
                add((32 * n * k + 4 * n * k + 4 * n * k // c["block"], 20 * n * k))
            else:
                kept = n * _kept(k, c["rate"])
                # four float32 arrays in, three out, the bf16 copy, flags, indices and packed values
                add((30 * n * k + n * k // c["block"] + 2 * kept + 4 * kept // c["block"], 16 * n * k))
    return {"bytes": total_bytes, "flops": total_flops}


def tolerance(case):
    kind = case["kind"]
    if kind in ("prune", "stack"):
        # float32 norms and a float64 sum of float32 terms; flags, indices, values and layouts are exact
        return {"rel": 1e-5, "max": 1e-4, "differ": 0.0}
    if kind in ("reweight", "retrain"):
        # float32 state; a bf16 copy may round the other way where the float32 value is near a tie
        return {"rel": 1e-4, "max": 8e-3, "differ": 1e-4}
    # bf16 outputs of float32 sums
    return {"rel": 4e-3, "max": 4e-2}
