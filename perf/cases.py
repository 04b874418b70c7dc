"""Performance cases of the library: what a program that serves Leech-lattice weights has it do.

A case is a dict of plain values; `prepare` makes what such a program holds before the call (records, scales,
activations, outputs, a captured graph where a serving loop would hold one), `run` is one pass through the public
entry points, `work` the bytes and operations the pass cannot do without.  Four kinds of pass:

  gemv     one matrix against one or several activation vectors, called directly (a plug-in, an evaluation loop).
  decode   a decoder's per-token sequence of row-concatenated launches (q+k+v, o, gate+up, down a layer), captured
           once as a CUDA graph and replayed every token; optionally on the rotated activation, with the FP16
           output head, or for a small batch of tokens (one launch a matrix: batched launches are not grouped).
  expand   block codes to records, at load time; the sparse overlay counts its exceptions first, to know that they fit.
  dequant  records to FP16 weights, the way to a library matrix product over a prompt (prefill).

Inputs are the synthetic stand-ins of the repository's own generator: a shell drawn uniformly, a point uniformly
inside it, fair gain bits, scales 0.02 |N(0, 1)|, activations N(0, 1), the in-dimension zero-padded to whole blocks.
"""
import torch

from paper_2609_02652_b200 import binding as B
from paper_2609_02652_b200 import datagen

LAYOUTS = {"planes": B.PLANES, "planes13": B.PLANES13, "planes10x": B.PLANES10X}
BLOCK_BYTES = {"planes": 14, "planes13": 13, "planes10x": 10}
VOCAB = 151936
MAX_LAUNCH_WEIGHTS = 36864 * 5120    # the largest launch of a matrix-vector product in the ranges below
MAX_MATRIX_WEIGHTS = 17408 * 5120    # the largest single matrix that is loaded or unpacked
ROTATION_BLOCK = 4096                # the longest rotation block the fused rotation always takes

_context = None


def context():
    """The process's one library context (tables and reduction scratch), as a serving process keeps it."""
    global _context
    if _context is None:
        _context = B.create(torch.cuda.current_device())
    return _context


def listed():
    return [
        # the smallest projection of a 4B-like decoder (k or v), called on its own: latency of one call
        {"name": "gemv_kv_1024x2560", "kind": "gemv", "layout": "planes", "rows": 1024, "k": 2560, "batch": 1},
        # a square projection of no particular model, odd in both directions (rows end inside a row group, leftover blocks)
        {"name": "gemv_odd_3071x3083", "kind": "gemv", "layout": "planes13", "rows": 3071, "k": 3083, "batch": 1},
        # the layout sweep's matrix: a large single launch
        {"name": "gemv_8192x8192", "kind": "gemv", "layout": "planes", "rows": 8192, "k": 8192, "batch": 1},
        # speculative or small-batch decode on one wide projection: eight activation vectors
        {"name": "gemv_batch8_4096x4096", "kind": "gemv", "layout": "planes", "rows": 4096, "k": 4096, "batch": 8},
        # one token through a 4B-like decoder layer, the launch-bound end of decode
        {"name": "decode_4b_layer", "kind": "decode", "layout": "planes", "hidden": 2560, "inter": 9728, "heads": 32, "kv_heads": 8,
         "layers": 1, "batch": 1, "rotate": False, "head": False},
        # the same layer in the smallest exact layout: a model that must leave room for a long cache
        {"name": "decode_4b_layer_overlay", "kind": "decode", "layout": "planes10x", "hidden": 2560, "inter": 9728, "heads": 32, "kv_heads": 8,
         "layers": 1, "batch": 1, "rotate": False, "head": False},
        # weights quantised in the rotated basis, as the paper's artifacts are: every launch rotates its activation
        {"name": "decode_8b_rotated", "kind": "decode", "layout": "planes", "hidden": 4096, "inter": 12288, "heads": 32, "kv_heads": 8,
         "layers": 2, "batch": 1, "rotate": True, "head": False},
        # four tokens at a time through an 8B-like layer
        {"name": "decode_8b_batch4", "kind": "decode", "layout": "planes", "hidden": 4096, "inter": 12288, "heads": 32, "kv_heads": 8,
         "layers": 1, "batch": 4, "rotate": False, "head": False},
        # one token through the whole 14B-like stack and the FP16 output head: the largest pass
        {"name": "decode_14b_stack_head", "kind": "decode", "layout": "planes", "hidden": 5120, "inter": 17408, "heads": 40, "kv_heads": 8,
         "layers": 40, "batch": 1, "rotate": False, "head": True},
        # loading: the codes of one feed-forward projection unfolded
        {"name": "expand_9728x2560", "kind": "expand", "layout": "planes", "rows": 9728, "k": 2560},
        # loading into the sparse overlay, a large projection: count, then expand
        {"name": "expand_overlay_17408x5120", "kind": "expand", "layout": "planes10x", "rows": 17408, "k": 5120},
        # prefill: one projection back to FP16 ahead of a library matrix product
        {"name": "dequant_4096x12288", "kind": "dequant", "layout": "planes", "rows": 4096, "k": 12288},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["gemv", "gemv", "decode", "decode", "expand", "dequant"])
    if kind == "decode":
        batch = rng.choice([1, 1, 1, 2, 4, 6])
        layout = "planes" if batch > 1 else rng.choice(["planes", "planes", "planes13", "planes10x"])
        heads = _log_uniform(rng, 8, 64)                         # head_dim 128 as in the 4B / 8B / 14B-like decoders
        hidden = 64 * _log_uniform(rng, 16, 96)                  # 1024 .. 6144; the attention width need not equal it
        return {"kind": "decode", "layout": layout, "hidden": hidden, "inter": 256 * _log_uniform(rng, 12, 72), "heads": heads,
                "kv_heads": min(heads, rng.choice([4, 8])), "layers": rng.randint(1, 4), "batch": batch,
                "rotate": layout == "planes" and batch == 1 and rng.random() < 0.4, "head": batch == 1 and rng.random() < 0.3}
    # projections from a k/v head group to a fused gate+up, any residue of rows and columns
    rows = _log_uniform(rng, 500, 36864 if kind == "gemv" else 17408)
    k = _log_uniform(rng, 1000, min(17408, (MAX_LAUNCH_WEIGHTS if kind == "gemv" else MAX_MATRIX_WEIGHTS) // rows))
    if kind == "gemv":
        batch = rng.choice([1, 1, 2, 3, 5, 8])
        layout = "planes" if batch > 1 else rng.choice(["planes", "planes13", "planes10x"])
        return {"kind": "gemv", "layout": layout, "rows": rows, "k": k, "batch": batch}
    if kind == "expand":
        return {"kind": "expand", "layout": rng.choice(["planes", "planes13", "planes10x"]), "rows": rows, "k": k}
    return {"kind": "dequant", "layout": "planes", "rows": rows, "k": k}


def _blocks_a_row(k):
    return (k + 23) // 24


def _launches(case):
    """The launches of one token as (in-dimension, [rows of each matrix]); the rows of a launch share their activation."""
    h, inter, q, kv = case["hidden"], case["inter"], 128 * case["heads"], 128 * case["kv_heads"]
    layer = [(h, [q, kv, kv]), (q, [h]), (h, [inter, inter]), (inter, [h])]
    if case["batch"] > 1:
        layer = [(k, [r]) for k, rows in layer for r in rows]
    return layer * case["layers"]


def _matrix(layout, rows, k, seed, tensor_id):
    """Records and row scales of one synthetic matrix, on the device."""
    nb = _blocks_a_row(k)
    codes = datagen.make_codes(rows, nb, seed, tensor_id, device="cuda")
    records = B.expand(context(), LAYOUTS[layout], codes, rows, nb)
    return records, datagen.make_row_scale(rows, seed, tensor_id).cuda()


def _activations(batch, k, seed, tensor_id):
    """Activation vectors padded to whole blocks: [k_padded], or [batch, k_padded] for more than one."""
    kp = 24 * _blocks_a_row(k)
    x = torch.stack([datagen.make_x(k, kp, seed, (tensor_id << 4) + j) for j in range(batch)])
    return (x if batch > 1 else x[0]).cuda()


def prepare(case, seed):
    if case["kind"] == "decode":
        return _prepare_decode(case, seed)
    rows, k = case["rows"], case["k"]
    nb = _blocks_a_row(k)
    state = {"case": case, "rows": rows, "nb": nb, "k_padded": 24 * nb, "layout": LAYOUTS[case["layout"]]}
    if case["kind"] == "expand":
        state["codes"] = datagen.make_codes(rows, nb, seed, device="cuda")
        if state["layout"] == B.PLANES10X:
            # the usual room for exceptions; the count says whether it is enough.  Zeroed: entries past the last exception
            # are not written
            state["out"] = torch.zeros(B.layout_bytes(B.PLANES10X, rows, 24 * nb), dtype=torch.uint8, device="cuda")
        return state
    state["records"], state["scale"] = _matrix(case["layout"], rows, k, seed, 0)
    if case["kind"] == "gemv":
        state["x"] = _activations(case["batch"], k, seed, 0)
    else:
        # the FP16 weights' buffer, which a prefill keeps and fills projection by projection
        state["W"] = torch.empty((rows, 24 * nb), dtype=torch.float16, device="cuda")
    return state


def _prepare_decode(case, seed):
    ctx, batch = context(), case["batch"]
    launches = _launches(case)
    # every output of the token in one buffer, launch by launch, [batch, rows] each
    y = torch.zeros(batch * sum(sum(rows) for _, rows in launches), dtype=torch.float32, device="cuda")
    calls, held, at, tensor_id = [], [y], 0, 0
    for k, rows_list in launches:
        x = _activations(batch, k, seed, tensor_id)
        problems = []
        for rows in rows_list:
            records, scale = _matrix(case["layout"], rows, k, seed, tensor_id)
            problems.append((records, scale, datagen.GAIN, y[at:at + batch * rows], rows))
            held += [records, scale]
            at += batch * rows
            tensor_id += 1
        held.append(x)
        calls.append(_call(case, ctx, problems, x, k))
    out = [y]
    if case["head"]:
        # the FP16 output head: random weights of a fan-in scale, the last hidden state as fp16
        generator = torch.Generator(device="cuda").manual_seed(seed)
        hidden = case["hidden"]
        W = torch.empty((VOCAB, hidden), dtype=torch.float16, device="cuda").normal_(0.0, hidden ** -0.5, generator=generator)
        xh = torch.empty((batch, hidden), dtype=torch.float16, device="cuda").normal_(0.0, 1.0, generator=generator)
        logits = torch.zeros((batch, VOCAB), dtype=torch.float32, device="cuda")
        held += [W, xh, logits]
        calls += [lambda j=j: B.gemv_fp16(W, xh[j], VOCAB, hidden, y=logits[j]) for j in range(batch)]
        out.append(logits)

    def token():
        for call in calls:
            call()

    token()                                      # warm-up; the first launch after an expansion is an ordinary one
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        token()
    return {"case": case, "graph": graph, "out": out, "held": held}


def _call(case, ctx, problems, x, k):
    """One launch of the token as a user's program issues it."""
    kp, layout = 24 * _blocks_a_row(k), LAYOUTS[case["layout"]]
    if case["batch"] > 1:
        records, scale, gain, y, rows = problems[0]
        return lambda: B.gemv_batch(ctx, records, scale, gain, x, rows, kp, y=y)
    array = B.make_problems(problems)
    if case["rotate"]:
        return lambda: B.gemv_rotated(ctx, array, x, kp, n=k, block=min(ROTATION_BLOCK, B.rotate_block(k)))
    return lambda: B.gemv_grouped(ctx, layout, array, x, kp)


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "decode":
        state["graph"].replay()
        return state["out"]
    ctx, rows, nb = context(), state["rows"], state["nb"]
    if kind == "gemv":
        if case["batch"] > 1:
            return B.gemv_batch(ctx, state["records"], state["scale"], datagen.GAIN, state["x"], rows, state["k_padded"])
        return B.gemv(ctx, state["layout"], state["records"], state["scale"], datagen.GAIN, state["x"], rows, state["k_padded"])
    if kind == "expand":
        if state["layout"] != B.PLANES10X:
            return B.expand(ctx, state["layout"], state["codes"], rows, nb)
        exceptions = B.overlay_count(ctx, state["codes"], rows, nb)
        if B.overlay_bytes(rows, 24 * nb, exceptions) > state["out"].numel():
            state["out"] = torch.zeros(B.overlay_bytes(rows, 24 * nb, exceptions), dtype=torch.uint8, device="cuda")
        return [exceptions, B.expand(ctx, state["layout"], state["codes"], rows, nb, out=state["out"])]
    return B.dequant_fp16(ctx, state["layout"], state["records"], state["scale"], datagen.GAIN, rows, state["k_padded"], W=state["W"])


def _gemv_work(layout, rows, k, batch):
    nb = _blocks_a_row(k)
    index = 4 * (-(-rows // 32)) * (nb // 4) if layout == "planes10x" else 0
    return BLOCK_BYTES[layout] * rows * nb + index + 2 * rows + batch * (48 * nb + 4 * rows), 2 * rows * k * batch


def work(case):
    if case["kind"] == "decode":
        total_bytes = flops = 0
        for k, rows_list in _launches(case):
            for rows in rows_list:
                b, f = _gemv_work(case["layout"], rows, k, case["batch"])
                total_bytes, flops = total_bytes + b, flops + f
            # the matrices of a launch share one activation
            total_bytes -= (len(rows_list) - 1) * case["batch"] * 48 * _blocks_a_row(k)
            if case["rotate"]:
                flops += k * (min(ROTATION_BLOCK, k & -k).bit_length() - 1)
        if case["head"]:
            total_bytes += 2 * VOCAB * case["hidden"] + case["batch"] * (2 * case["hidden"] + 4 * VOCAB)
            flops += 2 * VOCAB * case["hidden"] * case["batch"]
        return {"bytes": total_bytes, "flops": flops}
    rows, k, layout = case["rows"], case["k"], case["layout"]
    blocks = rows * _blocks_a_row(k)
    if case["kind"] == "gemv":
        total_bytes, flops = _gemv_work(layout, rows, k, case["batch"])
        return {"bytes": total_bytes, "flops": flops}
    if case["kind"] == "expand":
        return {"bytes": (8 + BLOCK_BYTES[layout]) * blocks, "flops": 0}
    return {"bytes": (14 + 48) * blocks + 2 * rows, "flops": 24 * blocks}


def tolerance(case):
    # records are integers written in a fixed order
    if case["kind"] == "expand":
        return "exact"
    # fp16(scale * gain / (4 sqrt m) * x_i), the product in f32: another order of the f32 factors moves a value that lies at
    # a rounding boundary by one fp16 unit, at most 2^-10 of it (4e-5 of 4e6 values against the f64 product: rel 7e-6)
    if case["kind"] == "dequant":
        return {"rel": 3e-5, "max": 1e-3}
    # f32 outputs.  Against the f64 sums of the same weights: rel 7e-8, max 6e-7 (the FP16 head: 2e-7, 9e-7); the same weights
    # summed by other f32 matrix-vector products: rel up to 4.1e-7, max up to 2.5e-6 (1024 x 2560 to 5120 x 17408)
    return {"rel": 1.6e-6, "max": 1e-5}
