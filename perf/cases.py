"""The work that users of this codec have it do, as cases that can be timed and compared.

A case is one call (a pass) through the public entry points of `paper_2410_16926_b200.pvq`, with
the count table and the amplitude codebook built beforehand, as a program that quantises more
than one matrix keeps them.  The listed cases are the workloads of `inputs.py` (and so of
`bench.py`), one direction at a time:

  - weights: encode once when a model is quantised, decode whenever it is used, a matrix at a time
    or all matrices of a decoder layer in one launch;
  - activations: quantised and dequantised on the fly (`roundtrip`), also straight from the
    unrotated values (`rotate_roundtrip`), with as many rows as there are tokens;

at the group sizes and code widths of the paper's tables: 16 values at 3 bits (the headline setting),
32 at 2 and 3 bits, 64 at 3 bits, 128 at 3 and 4 bits.  `draw` gives other row counts and row lengths
of the same operations, from a handful of tokens to whole layers, in both input types, and the
neighbouring settings (64 values at 4 bits, 256 at 3 bits, least-squares amplitudes).
"""
import math

import torch

from paper_2410_16926_b200 import pvq
from paper_2410_16926_b200.inputs import LLAMA3_8B_LAYER

# (group size, bits of a direction code, bits of an amplitude; 16: the amplitude itself as binary16)
WEIGHT_SETTINGS = ((16, 48, 4), (32, 64, 8), (32, 96, 4), (32, 96, 8), (64, 192, 6), (64, 256, 16), (128, 384, 16),
                   (256, 768, 16))
ACTIVATION_SETTINGS = ((32, 64, 8), (128, 512, 16))


def _case(op, rows, cols, setting, dtype="bf16", **more):
    group, bits, amp_bits = setting
    return dict(op=op, rows=rows, cols=cols, group=group, index_bits=bits, scale_bits=amp_bits, dtype=dtype, **more)


def listed():
    return [
        # the smallest matrix, fp32: what a call costs when there is next to no work in it
        dict(_case("encode", 512, 512, (32, 64, 8), "f32"), name="encode small fp32"),
        dict(_case("decode", 512, 512, (32, 64, 8)), name="decode small"),
        # one attention projection of an 8B model, quantised to 3.125 bits a weight
        dict(_case("encode", 4096, 4096, (32, 96, 4)), name="encode projection"),
        # the same projection at the paper's headline setting, read back
        dict(_case("decode", 4096, 4096, (16, 48, 4)), name="decode projection group 16"),
        # all seven matrices of a decoder layer in one launch: quantising a model, loading it
        dict(_case("encode_layer", 4096, 4096, (32, 96, 8), row_div=1), name="encode decoder layer"),
        dict(_case("decode_layer", 4096, 4096, (32, 96, 8), row_div=1), name="decode decoder layer"),
        # the largest single matrix of a 70B model, read back (codes of 192 bits)
        dict(_case("decode", 8192, 28672, (64, 192, 6)), name="decode 70B down projection"),
        # the weight-only setting of the paper's main table: group size 128, binary16 amplitudes
        dict(_case("encode", 4096, 4096, (128, 384, 16)), name="encode projection group 128"),
        dict(_case("decode", 4096, 4096, (128, 384, 16)), name="decode projection group 128"),
        # activations of a long prefill, quantised and dequantised on the fly
        dict(_case("roundtrip", 16384, 4096, (32, 64, 8)), name="activations"),
        # an ordinary prompt's activations, rotated on the fly first (an odd number of tokens)
        dict(_case("rotate_roundtrip", 1999, 4096, (32, 64, 8), block=4096), name="rotated activations"),
        # the paper's weight-and-activation setting: group size 128, 4 bits of direction a value
        dict(_case("roundtrip", 16384, 4096, (128, 512, 16)), name="activations group 128"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("encode", "encode", "decode", "decode", "encode_layer", "decode_layer", "roundtrip", "roundtrip",
                     "rotate_roundtrip"))
    dtype = "f32" if rng.random() < 0.2 else "bf16"
    if op in ("encode_layer", "decode_layer"):  # a layer of the same model, or a slice of its rows (tensor parallel)
        return _case(op, 4096, 4096, rng.choice(((16, 48, 4), (32, 64, 8), (32, 96, 4), (32, 96, 8), (64, 192, 6))),
                     row_div=rng.choice((1, 2, 3, 4, 5, 7, 8, 13, 16)))
    if op in ("encode", "decode"):
        setting = rng.choice(WEIGHT_SETTINGS)
        group = setting[0]
        heavy = group > 64 or setting[1] > 32 * 6
        least_squares = op == "encode" and rng.random() < 0.15
        cols = group * max(2, round(_log_uniform(rng, 512, 28672) / group))
        if heavy or least_squares:  # encoding keeps a whole row of these in one thread block
            cols = min(cols, group * (128 if heavy else 448))
        most = (1 << (25 if heavy else 27)) // (2 if dtype == "f32" else 1)
        rows = max(1, min(_log_uniform(rng, 64, 16384), most // cols))
        if op == "decode":
            return _case(op, rows, cols, setting)
        return _case(op, rows, cols, setting, dtype, least_squares=least_squares)
    setting = rng.choice(ACTIVATION_SETTINGS)
    tokens = _log_uniform(rng, 1, 8192)
    if op == "roundtrip":
        cols = setting[0] * max(2, round(_log_uniform(rng, 512, 8192) / setting[0]))
        return _case(op, tokens, cols, setting, dtype)
    block = rng.choice((512, 1024, 2048, 4096))
    cols = block * rng.randint(1, 8192 // block)
    tokens = min(tokens, (1 << 25) // cols)
    return _case(op, tokens, cols, setting, dtype, block=block)


def _rotate(x, block, signs):
    """x (fp32, rows x cols) with every run of `block` columns multiplied by signs and H / sqrt(block)."""
    rows, cols = x.shape
    y = x.view(rows, cols // block, block) * signs
    h = 1
    while h < block:
        y = y.view(rows, cols // block, block // (2 * h), 2, h)
        y = torch.cat((y[:, :, :, :1] + y[:, :, :, 1:], y[:, :, :, :1] - y[:, :, :, 1:]), dim=3)
        h *= 2
    return y.reshape(rows, cols) * (1.0 / math.sqrt(block))


def _gaussian(gen, *shape):
    return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32)


def _weights(gen, rows, cols, dtype):
    """Rotated weights: heavy-tailed entries (Student's t with 5 degrees of freedom) of scale 0.02, then
    a random-sign Hadamard on blocks of the largest power of two up to 512 that divides the rows."""
    out = torch.empty((rows, cols), device="cuda", dtype=dtype)
    block = min(512, cols & -cols)
    signs = torch.where(torch.rand(block, generator=gen, device="cuda") < 0.5, -1.0, 1.0)
    step = max(1, (1 << 24) // cols)
    for r in range(0, rows, step):
        n = min(step, rows - r)
        chi = sum(_gaussian(gen, n, cols).square_() for _ in range(5)) / 5
        x = _gaussian(gen, n, cols) * 0.02 / chi.sqrt_()
        out[r:r + n] = _rotate(x, block, signs)
    return out


def _activations(gen, rows, cols, dtype, rotated):
    """Rows of N(0,1) with one channel in a thousand 20 times larger; `rotated`: already multiplied by
    a random-sign Hadamard on blocks of the largest power of two up to 4096 that divides the rows."""
    x = _gaussian(gen, rows, cols)
    channels = torch.randperm(cols, generator=gen, device="cuda")[:max(1, round(cols * 0.001))]
    x[:, channels] *= 20.0
    if rotated:
        block = min(4096, cols & -cols)
        signs = torch.where(torch.rand(block, generator=gen, device="cuda") < 0.5, -1.0, 1.0)
        step = max(1, (1 << 24) // cols)
        for r in range(0, rows, step):
            x[r:r + step] = _rotate(x[r:r + step], block, signs)
    return x.to(dtype)


def _matrices(case):
    """[(rows, cols)] of the case: one matrix, or those of a decoder layer."""
    if case["op"].endswith("_layer"):
        return [(max(1, r // case["row_div"]), c) for _, r, c in LLAMA3_8B_LAYER]
    return [(case["rows"], case["cols"])]


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    op, N, b = case["op"], case["group"], case["scale_bits"]
    dtype = torch.float32 if case["dtype"] == "f32" else torch.bfloat16
    K = pvq.max_pulses(N, case["index_bits"])
    state = dict(op=op, N=N, K=K, b=b, dtype=dtype, table=pvq.build_count_table(N, K),
                 amp_mode=1 if case.get("least_squares") else None)
    books = {}

    def book(cols):
        if b == 16:
            return None, None
        if cols not in books:
            books[cols] = pvq.build_scale_codebook(N, cols // N, b)
        return books[cols]

    if op in ("roundtrip", "rotate_roundtrip"):
        state["x"] = _activations(gen, case["rows"], case["cols"], dtype, op == "roundtrip")
        state["edges"], state["levels"] = book(case["cols"])
        if op == "rotate_roundtrip":
            state["block"] = case["block"]
            state["signs"] = torch.where(torch.rand(case["block"], generator=gen, device="cuda") < 0.5, -1.0, 1.0)
        return state
    items = []
    for rows, cols in _matrices(case):
        edges, levels = book(cols)
        x = _weights(gen, rows, cols, dtype)
        if op == "encode":
            state.update(x=x, edges=edges)
            return state
        if op == "decode":
            codes, scale_idx, row_norm = pvq.encode(x, N, K, b, state["table"], edges)
            state.update(codes=codes, scale_idx=scale_idx, row_norm=row_norm, levels=levels)
            return state
        codes, scale_idx, row_norm = pvq.alloc_encoded(rows, cols // N, pvq.code_words(N, K), b)
        item = dict(codes=codes, scale_idx=scale_idx, row_norm=row_norm, edges=edges, levels=levels, cols=cols)
        if op == "decode_layer":
            pvq.encode(x, N, K, b, state["table"], edges, out=(codes, scale_idx, row_norm))
            item["out"] = torch.empty((rows, cols), dtype=torch.bfloat16, device="cuda")
        else:
            item["x"] = x
        items.append(item)
    state["items"] = items
    return state


def run(state):
    s = state
    op, N, K, b, table = s["op"], s["N"], s["K"], s["b"], s["table"]
    if op == "encode":
        return pvq.encode(s["x"], N, K, b, table, s["edges"], amp_mode=s["amp_mode"])
    if op == "decode":
        return pvq.decode(s["codes"], s["scale_idx"], s["row_norm"], N, K, b, table, s["levels"])
    if op == "roundtrip":
        return pvq.roundtrip(s["x"], N, K, b, table, s["edges"], s["levels"])
    if op == "rotate_roundtrip":
        return pvq.rotate_roundtrip(s["x"], s["block"], s["signs"], N, K, b, table, s["edges"], s["levels"])
    if op == "encode_layer":
        pvq.encode_batched(s["items"], s["dtype"], N, K, b, table)
        return [(it["codes"], it["scale_idx"], it["row_norm"]) for it in s["items"]]
    pvq.decode_batched(s["items"], N, K, b, table)
    return [it["out"] for it in s["items"]]


def work(case):
    """Bytes: the values, the codes (as the words they are stored in), the amplitudes and the row norms, each once.
    Operations: those on the values that any way of computing the result shares (encoding: the two norms,
    scaling, floor and residual; decoding: the sum of squares and the scaling; 2 log2(block) / 2 for a
    rotation), not the integer arithmetic of the codes."""
    op, N, b = case["op"], case["group"], case["scale_bits"]
    words = (case["index_bits"] + 31) // 32
    in_bytes = 4 if case["dtype"] == "f32" else 2
    total = {"bytes": 0, "flops": 0}
    for rows, cols in _matrices(case):
        G = cols // N
        values = rows * cols
        packed = rows * G * words * 4 + rows * ((G * b + 31) // 32) * 4 + (rows * 4 if op.startswith("encode") or b != 16 else 0)
        if op.startswith("encode"):
            total["bytes"] += values * in_bytes + packed
            total["flops"] += 6 * values
        elif op.startswith("decode"):
            total["bytes"] += packed + values * 2
            total["flops"] += 3 * values
        else:
            total["bytes"] += values * in_bytes + values * 2
            total["flops"] += 9 * values
            if op == "rotate_roundtrip":
                total["flops"] += values * (int(math.log2(case["block"])) + 1)
    return total


def tolerance(case):
    # Codes, amplitude indices and norms are fixed by the stated arithmetic, and the decoded values
    # are bf16 roundings of fp32 products of them: nothing is left open.
    return "exact"
