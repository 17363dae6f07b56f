"""The work that is timed: what programs have this library do, through its public calls.

A case is a dict of plain values.  `kind` says which calls one pass makes:

  prefill   pa_prefill over a kept layout (`layout` "kept": every layer of a model shares it) or
            pa_build_layout + pa_prefill ("built": the first layer of a prompt of a new length);
            `block` above 64: the mask's block, listed in 64-token tiles
  varlen    pa_prefill_varlen over prompts of different lengths packed into one tensor
  train     pa_prefill + pa_prefill_backward: O, LSE, dQ, dK, dV of one layer
  decode    pa_decode against a contiguous cache
  paged     pa_decode_paged against a pool of 64-token pages in scrambled order
  steps     several decoding steps of a paged batch: pa_kv_append + pa_decode_paged each

`seq` is the length (varlen and the decode kinds: the longest), `min_seq` the shortest one where the
sequences differ; the lengths follow from the case, all other inputs from the seed.  Shapes are those of
the repository's workloads and tests (28 query heads on 4 KV heads of 128 features and smaller ones);
tensors are N(0, 1) rounded to bf16 as in synth_inputs.py, K times `k_scale`.
"""
import math
import random

import torch

import paper_2503_03588_b200 as pa
from paper_2503_03588_b200.binding import decode_params, paged_params


def _case(name, kind, seq, batch=1, heads=(28, 4, 128), window=5, sink=1, block=64, k_scale=1.0, layout="kept",
          out="bf16", min_seq=0, steps=0):
    hq, hkv, d = heads
    c = {"kind": kind, "batch": batch, "seq": seq, "min_seq": min_seq or seq, "q_heads": hq, "kv_heads": hkv,
         "head_dim": d, "window": window, "sink": sink, "block": block, "k_scale": k_scale, "layout": layout,
         "out": out, "steps": steps}
    return dict(c, name=name) if name else c


def listed():
    return [
        # One user's token against a short chat: nothing but latency.
        _case("decode_b1_4k", "decode", 4001),
        # The decode benchmark: eight long contexts, 64K to 128K tokens.
        _case("decode_b8_128k", "decode", 131072, batch=8, min_seq=65536),
        # A full serving batch on a paged cache: bandwidth.
        _case("decode_paged_b256_16k", "paged", 16384, batch=256, min_seq=4096),
        # Generation: 16 tokens for each of eight sequences behind a 16K context, append + decode per step.
        _case("decode_steps_b8_16k", "steps", 16384, batch=8, min_seq=15000, steps=16),
        # The smallest prefill configuration: 2 heads of 64 features, window 1.
        _case("prefill_2k_d64", "prefill", 2048, heads=(2, 2, 64), window=1),
        # The 32K benchmark prompt, peaky logits.
        _case("prefill_32k_peaky", "prefill", 32768, k_scale=3.0),
        # The 128K benchmark prompt, layout included.
        _case("prefill_128k_built", "prefill", 131072, layout="built"),
        # Prompts of several users packed into one call.
        _case("prefill_varlen_8x12k", "varlen", 12000, batch=8, min_seq=300),
        # The mask in the paper's own 256-token blocks, a ragged length.
        _case("prefill_16k_block256", "prefill", 16100, block=256),
        # Fine-tuning on short samples: forward and backward, a ragged length.
        _case("train_4k", "train", 4001),
        # Long-context training: forward and backward at 32K.
        _case("train_32k", "train", 32768),
        # Training a small model: heads of 64 features, batch 2.
        _case("train_8k_d64", "train", 8192, batch=2, heads=(16, 4, 64)),
    ]


_HEADS_128 = [(28, 4, 128)] * 3 + [(14, 2, 128), (8, 2, 128), (16, 2, 128), (7, 1, 128), (8, 8, 128)]
_HEADS_64 = [(16, 4, 64), (8, 2, 64), (8, 8, 64), (2, 2, 64)]


def _size(rng, lo, hi):
    """Log-uniform in [lo, hi]; one in four a multiple of 64, the others as they fall."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, n // 64 * 64 if rng.random() < 0.25 else n))


def draw(rng):
    kind = rng.choice(["decode", "paged", "steps", "prefill", "prefill", "varlen", "train", "train"])
    heads = rng.choice(_HEADS_128 if rng.random() < 0.75 else _HEADS_64)
    window, sink = rng.choice([(5, 1), (5, 1), (5, 1), (9, 1), (1, 1), (3, 2)])
    more = {"window": window, "sink": sink, "heads": heads, "k_scale": rng.choice([1.0, 1.0, 2.0, 3.0])}
    if kind in ("decode", "paged"):
        seq = _size(rng, 200, 131072)
        batch = _size(rng, 1, 256)
        while batch > 1 and batch * seq * heads[1] * heads[2] > 256 * 16384 * 512:  # the listed batch's cache
            batch //= 2
        return _case(None, kind, seq, batch=batch, min_seq=max(1, seq // rng.choice([1, 2, 8])), **more)
    if kind == "steps":
        seq = _size(rng, 500, 32768)
        return _case(None, kind, seq, batch=_size(rng, 1, 32), min_seq=max(1, seq // 2), steps=rng.randint(4, 16), **more)
    if kind == "train":
        seq = _size(rng, 500, 32768 if heads[2] == 128 else 8192)
        batch = rng.choice([1, 1, 2, 3])
        while batch > 1 and batch * seq * heads[0] * heads[2] > 32768 * 28 * 128 // (1 if heads[2] == 128 else 4):
            batch -= 1
        return _case(None, kind, seq, batch=batch, **more)
    more["out"] = "f32" if rng.random() < 0.15 else "bf16"
    if kind == "varlen":
        seq = _size(rng, 300, 32768)
        batch = rng.randint(2, 12)
        while batch > 2 and batch * seq > 100000:
            batch -= 1
        return _case(None, kind, seq, batch=batch, min_seq=max(1, seq // 40), **more)
    block = 256 if rng.random() < 0.25 else 64
    seq = _size(rng, 200, 131072 if block == 64 else 32768)
    batch = rng.choice([1, 1, 2, 4])
    while batch > 1 and batch * seq > (131072 if block == 64 else 32768):
        batch //= 2
    return _case(None, kind, seq, batch=batch, block=block, layout=rng.choice(["kept", "built"]), **more)


def _lens(case):
    """The sequences' lengths (decode: cached tokens, the current one included)."""
    rng = random.Random("%d %d %d" % (case["batch"], case["seq"], case["min_seq"]))
    return [case["seq"]] + [rng.randint(case["min_seq"], case["seq"]) for _ in range(case["batch"] - 1)]


class _Draws:
    """bf16 N(0, 1) tensors from one seed, drawn on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device="cuda").manual_seed(seed)

    def __call__(self, *shape, scale=1.0):
        t = torch.randn(shape, generator=self.g, device="cuda", dtype=torch.bfloat16)
        return t.mul_(scale) if scale != 1.0 else t


def _layout(case):
    if case["block"] == 64:
        return pa.pa_build_layout(case["seq"], 64, case["window"], case["sink"])
    return pa.pa_build_tile_layout(case["seq"], case["block"], case["window"], case["sink"], 64)


def prepare(case, seed):
    draw_ = _Draws(seed)
    b, n, hq, hkv, d = (case[k] for k in ("batch", "seq", "q_heads", "kv_heads", "head_dim"))
    s = {"case": case, "dtype": torch.float32 if case["out"] == "f32" else torch.bfloat16}
    kind = case["kind"]
    if kind in ("prefill", "train"):
        s["q"], s["k"], s["v"] = draw_(b, n, hq, d), draw_(b, n, hkv, d, scale=case["k_scale"]), draw_(b, n, hkv, d)
        if kind == "train":
            s["d_o"] = draw_(b, n, hq, d)
        if case["layout"] == "kept":
            s["layout"] = _layout(case)
        return s
    lens = _lens(case)
    if kind == "varlen":
        cu = [0]
        for x in lens:
            cu.append(cu[-1] + x)
        s["q"], s["k"], s["v"] = draw_(cu[-1], hq, d), draw_(cu[-1], hkv, d, scale=case["k_scale"]), draw_(cu[-1], hkv, d)
        s["cu"] = torch.tensor(cu, dtype=torch.int32, device="cuda")
        s["layout"] = _layout(case)
        return s
    # A decode loop keeps its outputs and scratch.
    s["lens"] = torch.tensor(lens, dtype=torch.int32, device="cuda")
    steps = max(1, case["steps"])
    s["q"] = [draw_(b, hq, d) for _ in range(steps)]
    s["o"] = torch.empty((steps, b, hq, d), dtype=s["dtype"], device="cuda")
    s["lse"] = torch.empty((steps, b, hq), dtype=torch.float32, device="cuda")
    s["o_t"], s["lse_t"] = list(s["o"].unbind(0)), list(s["lse"].unbind(0))
    if kind == "decode":
        s["k"], s["v"] = draw_(b, n, hkv, d, scale=case["k_scale"]), draw_(b, n, hkv, d)
        params = decode_params(s["q"][0], s["k"], s["v"], case["window"], case["sink"], o_dtype=s["dtype"])
        s["ws"] = torch.empty(pa.pa_decode_workspace_bytes(params), dtype=torch.uint8, device="cuda")
        return s
    blocks = (n + case["steps"] + 63) // 64
    s["k"], s["v"] = draw_(b * blocks, 64, hkv, d, scale=case["k_scale"]), draw_(b * blocks, 64, hkv, d)
    order = torch.randperm(b * blocks, generator=draw_.g, device="cuda")
    s["table"] = order.to(torch.int32).view(b, blocks).contiguous()
    params = paged_params(s["q"][0], s["k"], s["v"], s["table"], case["window"], case["sink"], o_dtype=s["dtype"])
    s["ws"] = torch.empty(pa.pa_decode_paged_workspace_bytes(params), dtype=torch.uint8, device="cuda")
    if kind == "steps":
        s["context"] = s["lens"].clone()
        s["k_new"] = [draw_(b, hkv, d, scale=case["k_scale"]) for _ in range(steps)]
        s["v_new"] = [draw_(b, hkv, d) for _ in range(steps)]
    return s


def run(s):
    case = s["case"]
    kind, window, sink = case["kind"], case["window"], case["sink"]
    if kind == "prefill":
        built = case["layout"] == "built"
        row_ptr, col_idx = _layout(case) if built else s["layout"]
        o, lse, _ = pa.pa_prefill(s["q"], s["k"], s["v"], row_ptr, col_idx, o_dtype=s["dtype"])
        return (o, lse, row_ptr, col_idx) if built else (o, lse)
    if kind == "train":
        row_ptr, col_idx = s["layout"]
        o, lse, _ = pa.pa_prefill(s["q"], s["k"], s["v"], row_ptr, col_idx)
        dq, dk, dv, _ = pa.pa_prefill_backward(s["q"], s["k"], s["v"], o, lse, s["d_o"], row_ptr, col_idx)
        return o, lse, dq, dk, dv
    if kind == "varlen":
        o, lse, _ = pa.pa_prefill_varlen(s["q"], s["k"], s["v"], s["cu"], case["seq"], *s["layout"], o_dtype=s["dtype"])
        return o, lse
    if kind == "decode":
        pa.pa_decode(s["q"][0], s["k"], s["v"], s["lens"], window, sink, o=s["o_t"][0], lse=s["lse_t"][0],
                     workspace=s["ws"])
        return s["o"], s["lse"]
    if kind == "paged":
        pa.pa_decode_paged(s["q"][0], s["k"], s["v"], s["table"], s["lens"], window, sink, o=s["o_t"][0],
                           lse=s["lse_t"][0], workspace=s["ws"])
        return s["o"], s["lse"]
    # steps: a request starts from its context and grows by one token per step
    s["lens"].copy_(s["context"])
    for t in range(case["steps"]):
        pa.pa_kv_append(s["k_new"][t], s["v_new"][t], s["k"], s["v"], s["table"], s["lens"])
        pa.pa_decode_paged(s["q"][t], s["k"], s["v"], s["table"], s["lens"], window, sink, o=s["o_t"][t], lse=s["lse_t"][t],
                           workspace=s["ws"])
    return s["o"], s["lse"], s["k"], s["v"], s["lens"]


def _row_blocks(i, window, sink):
    """How many key blocks query block i lists (distances below the window, powers of two, sink blocks)."""
    w = max(window, 1)
    n = min(i + 1, w) + max(0, min(sink, i - w + 1))
    step = 1
    while step <= i:
        if step >= w and i - step >= sink:
            n += 1
        step *= 2
    return n


def _pairs(n, block, window, sink):
    """Attended (query, key) token pairs of one head of a sequence of n tokens."""
    total = 0
    for i in range((n + block - 1) // block):
        rows = min(block, n - i * block)
        total += (_row_blocks(i, window, sink) - 1) * block * rows + rows * (rows + 1) // 2
    return total


def work(case):
    b, hq, hkv, d = (case[k] for k in ("batch", "q_heads", "kv_heads", "head_dim"))
    window, sink, kind = case["window"], case["sink"], case["kind"]
    o_bytes = 4 if case["out"] == "f32" else 2
    if kind in ("prefill", "varlen", "train"):
        lens = _lens(case) if kind == "varlen" else [case["seq"]] * b
        tokens = sum(lens)
        pairs = sum(_pairs(n, case["block"], window, sink) for n in (lens if kind == "varlen" else lens[:1]))
        pairs *= 1 if kind == "varlen" else b
        # Q, K, V in; O and LSE out.  Two products forward.
        size = tokens * (hq * d * (2 + o_bytes) + 2 * hkv * d * 2 + hq * 4)
        flops = 4 * pairs * hq * d
        if kind == "train":  # dO in; dQ, dK, dV out in fp32 (Q, K, V, O are there already).  Five products.
            size += tokens * (hq * d * (2 + 4) + 2 * hkv * d * 4)
            flops += 10 * pairs * hq * d
        return {"bytes": size, "flops": flops}
    size = flops = 0
    for t in range(max(1, case["steps"])):
        for n in _lens(case):
            n += t + 1 if kind == "steps" else 0
            keys = (_row_blocks((n - 1) // 64, window, sink) - 1) * 64 + (n - 1) % 64 + 1
            size += keys * hkv * d * 2 * 2 + hq * (d * (2 + o_bytes) + 4)
            flops += 4 * keys * hq * d
            if kind == "steps":
                size += 2 * 2 * hkv * d * 2
    return {"bytes": size, "flops": flops}


def tolerance(case):
    # bf16 operands and bf16 P (and dS) between the two products, fp32 sums.  Against fp64 on up to 4001 tokens:
    # O and LSE 2.2e-3 and at most 0.025 of the larger of the value and the root mean square, gradients 3.0e-3
    # and 0.12 (rows whose dO O almost cancels); stated at four times that.
    return {"rel": 1.2e-2, "max": 0.5} if case["kind"] == "train" else {"rel": 9e-3, "max": 0.1}
