"""Performance cases of the PM-KVQ cache: the calls that a serving or calibration program makes, over the range of sizes
it makes them at.

Five kinds of work:

  decode      a whole-model decode loop: ``Cache.decode_step`` (append + eviction + attention of every block) for a few
              tokens in a row on a warm cache.  Every pass continues the same context; the roll-back between passes
              (``restore_layer_state``, host side only) is what a program does that samples several continuations of one
              prefix or drops rejected draft tokens.
  layerwise   the same token loop the way an engine drives it whose next block's Keys need the previous block's output:
              ``append`` and ``decode_attention`` block by block.
  prefill     a prompt written into an empty cache (one ``append`` per block) and the first decode step behind it.
  chunked     a long context written in chunks, through the progressive 16 -> 8 -> 4 -> 2 reduces that its budgets ask for,
              and the first decode step behind it.
  calibrate   ``calibrate_lambda``: the equalization vector of one block from calibration Keys.
  alpha_grid  ``alpha_grid_search``: the exponent of the equalization vector on one block's calibration tensors.

Shapes are those of the 7B / 8B / 32B / 70B workloads of this repository's benchmark (28 Q / 4 KV, 32 / 8, 40 / 8 and 64 / 8
heads, 32K to 128K maximum context, Fbit 2 and 4), with the number of blocks cut where a whole model would not fit three
times, plus the one-block 4 Q / 1 KV case of its parity tests.  The width of a cache's body is what the policy gives at that
context length.  All caches use the default contraction path; the other one (``attention_path = 1``) is documented as
the slower one, so no program picks it.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2505_18610_b200 import synth
from paper_2505_18610_b200.binding import Cache, alpha_grid_search, calibrate_lambda

N_SINK, WINDOW = 1, 128
N_OUTLIER, OUTLIER_FACTOR = 4, 15.0
DEVICE = "cuda"

# what a drawn case may cost at most: below the largest listed ones
MOST_BYTES = 5.5e9       # bytes one pass reads and writes
MOST_FLOPS = 3.5e12      # of an alpha grid search


def listed():
    return [
        # the smallest job there is: one block, one sequence, a 4K context at its final 4 bit; all latency
        dict(name="decode_1block_b1_4k", kind="decode", layers=1, q_heads=4, kv_heads=1, batch=1, context=4085,
             max_tokens=4096, edge_bits=4, inner_bits=4, evict_chunk=1, steps=4),
        # one user in front of a 7B model early in a generation: every block still at 16 bit
        dict(name="decode_7b_b1_3k", kind="decode", layers=28, q_heads=28, kv_heads=4, batch=1, context=3001,
             max_tokens=32768, edge_bits=4, inner_bits=2, evict_chunk=1, steps=4),
        # a small batch in mid-generation: blocks at 8 and 4 bit
        dict(name="decode_7b_b4_11k", kind="decode", layers=28, q_heads=28, kv_heads=4, batch=4, context=11003,
             max_tokens=32768, edge_bits=4, inner_bits=2, evict_chunk=1, steps=4),
        # uniform 4 bit, evictions in groups of 16
        dict(name="decode_8b_b8_20k", kind="decode", layers=16, q_heads=32, kv_heads=8, batch=8, context=20011,
             max_tokens=32768, edge_bits=4, inner_bits=4, evict_chunk=16, steps=4),
        # the long end of a generation at full batch: 20 blocks at 2 bit, 8 at 4 bit, the benchmark's own shape
        dict(name="decode_7b_b16_32k", kind="decode", layers=28, q_heads=28, kv_heads=4, batch=16, context=32760,
             max_tokens=32768, edge_bits=4, inner_bits=2, evict_chunk=1, steps=2),
        # block-by-block engine, small batch, 16 bit
        dict(name="layerwise_32b_b2_9k", kind="layerwise", layers=16, q_heads=40, kv_heads=8, batch=2, context=9001,
             max_tokens=131072, edge_bits=4, inner_bits=2, evict_chunk=1, steps=2),
        # block-by-block engine at the long end: group of 8 query heads, 2 bit
        dict(name="layerwise_70b_b16_64k", kind="layerwise", layers=4, q_heads=64, kv_heads=8, batch=16, context=65500,
             max_tokens=65536, edge_bits=2, inner_bits=2, evict_chunk=1, steps=2),
        # an ordinary prompt, one sequence, ragged length
        dict(name="prefill_7b_b1_2537", kind="prefill", layers=28, q_heads=28, kv_heads=4, batch=1, context=2537,
             max_tokens=32768, edge_bits=4, inner_bits=2, evict_chunk=1),
        # long prompts, a small batch
        dict(name="prefill_8b_b4_8k", kind="prefill", layers=8, q_heads=32, kv_heads=8, batch=4, context=8192,
             max_tokens=32768, edge_bits=4, inner_bits=4, evict_chunk=1),
        # a whole context in chunks of 2048, through every progressive reduce
        dict(name="chunked_7b_b8_32k", kind="chunked", layers=2, q_heads=28, kv_heads=4, batch=8, context=32760,
             max_tokens=32768, edge_bits=2, inner_bits=2, evict_chunk=1, chunk=2048),
        # calibration Keys of one block: 128 samples of 2048 tokens, positions interpolated by 4
        dict(name="calibrate_8b_2k_x128", kind="calibrate", tokens=2048, sequences=128, kv_heads=8, pos_scale=4.0),
        # alpha of one 7B block: two samples of 2048 tokens, the 20-point grid, the loss at 2 bit
        dict(name="alpha_grid_7b_2k_x2", kind="alpha_grid", tokens=2048, sequences=2, kv_heads=4, group=7, bits=2,
             alphas=20, pos_scale=4.0),
    ]


# query heads, KV heads, blocks, Fbit of the outer and of the inner blocks, maximum contexts
MODELS = [
    (28, 4, 28, 4, 2, (32768,)),
    (32, 8, 32, 4, 4, (32768,)),
    (40, 8, 32, 4, 2, (32768, 131072)),
    (64, 8, 16, 2, 2, (32768, 65536)),
    (4, 1, 1, 4, 4, (4096, 32768)),
    (8, 2, 2, 4, 2, (2048, 16384)),
]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode"] * 5 + ["layerwise"] * 2 + ["prefill"] * 2 + ["chunked", "calibrate", "alpha_grid"])
    while True:
        if kind == "calibrate":
            case = dict(kind=kind, tokens=_log_int(rng, 200, 4096), sequences=_log_int(rng, 1, 128),
                        kv_heads=rng.choice([1, 2, 4, 8]), pos_scale=rng.choice([1.0, 4.0]))
        elif kind == "alpha_grid":
            kv_heads, group = rng.choice([(4, 7), (8, 4), (8, 5), (8, 8), (1, 4)])
            case = dict(kind=kind, tokens=_log_int(rng, 250, 2048), sequences=rng.randint(1, 3), kv_heads=kv_heads,
                        group=group, bits=rng.choice([2, 2, 4]), alphas=rng.choice([10, 20]),
                        pos_scale=rng.choice([1.0, 4.0]))
        else:
            q_heads, kv_heads, layers, edge, inner, maxima = rng.choice(MODELS)
            max_tokens = rng.choice(maxima)
            layers = rng.randint(1, layers)
            case = dict(kind=kind, layers=layers, q_heads=q_heads, kv_heads=kv_heads, batch=_log_int(rng, 1, 32),
                        context=_log_int(rng, 300, max_tokens - 8), max_tokens=max_tokens, edge_bits=edge, inner_bits=inner,
                        evict_chunk=rng.choice([1, 1, 1, 8, 16]))
            if kind in ("decode", "layerwise"):
                case["steps"] = rng.randint(1, 4)
                if kind == "layerwise":
                    case["layers"] = min(layers, 16)
            elif kind == "prefill":
                case["layers"], case["context"] = min(layers, 16), min(case["context"], 16000)
            else:
                case["layers"], case["chunk"] = min(layers, 2), rng.choice([512, 1000, 2048, 4096])
        w = work(case)
        if w["bytes"] <= MOST_BYTES and (kind != "alpha_grid" or w["flops"] <= MOST_FLOPS) and _footprint(case) <= 16e9:
            return case


# ---- sizes -----------------------------------------------------------------------------------------------------------

def _fbits(case):
    return synth.bit_schedule(case["layers"], case["edge_bits"], case["inner_bits"])


def _body(case, n):
    return max(0, (n - N_SINK - WINDOW) // case["evict_chunk"] * case["evict_chunk"])


def _token_bytes(case, n, bits):
    """Bytes of one slice's n cached tokens, K and V: codes, fp32 scale, fp32 zero-point."""
    body = _body(case, n)
    return 2 * ((n - body) * (16 * 16 + 8) + body * (16 * bits + 8))


def _width(case, fbit, n):
    """Width the policy leaves a block's body at once it holds n tokens: the default budget is the block's size with
    max_tokens tokens and the body at Fbit."""
    m, c = case["max_tokens"], case["evict_chunk"]
    budget = max(_token_bytes(case, k, fbit) for k in range(max(0, m - c + 1), m + 1))
    bits = 16
    while bits > fbit and _token_bytes(case, n, bits) > budget:
        bits //= 2
    return bits


def _footprint(case):
    """Device bytes of one state, roughly."""
    if case["kind"] in ("calibrate", "alpha_grid"):
        return work(case)["bytes"] * 8
    slices = case["batch"] * case["kv_heads"]
    cache = sum(slices * _token_bytes(case, case["max_tokens"], f) for f in _fbits(case))
    given = case["context"] if case["kind"] in ("prefill", "chunked") else 0
    return cache + case["layers"] * slices * given * 512


def work(case):
    if case["kind"] == "calibrate":
        n = case["tokens"] * case["sequences"] * case["kv_heads"]
        return {"bytes": n * 256 + case["kv_heads"] * 512, "flops": n * 128 * 3}
    if case["kind"] == "alpha_grid":
        n, heads = case["tokens"], case["kv_heads"] * case["group"]
        vectors = n * case["sequences"] * (2 * case["kv_heads"] + heads)
        pairs = n * (n + 1) // 2 * case["sequences"] * heads
        return {"bytes": vectors * 256 + 8 * case["alphas"], "flops": (case["alphas"] + 1) * pairs * 512}
    slices, layers = case["batch"] * case["kv_heads"], case["layers"]
    q_vectors = layers * case["batch"] * case["q_heads"]
    prompt = case["context"] if case["kind"] in ("prefill", "chunked") else 0
    total = flops = 0
    if prompt:                       # the prompt's K and V in, its codes out
        total += layers * slices * prompt * 512
        total += sum(slices * _token_bytes(case, prompt, _width(case, f, prompt)) for f in _fbits(case))
    for step in range(case.get("steps", 1)):
        n = case["context"] + step + 1
        total += sum(slices * _token_bytes(case, n, _width(case, f, n)) for f in _fbits(case))    # attention reads the cache
        total += layers * slices * (512 + 528) + q_vectors * 128 * (2 + 4)                        # new token; Q in, output
        total += layers * case["kv_heads"] * 512
        flops += q_vectors * n * 512
    return {"bytes": total, "flops": flops}


def tolerance(case):
    if case["kind"] == "calibrate":
        return {"rel": 1e-5, "max": 2e-5}      # an fp32 rotation and a power
    if case["kind"] == "alpha_grid":
        return {"rel": 2e-3, "max": 5e-3}      # small differences of two attention outputs, 22-bit operands
    # attention over quantized tokens, probabilities carried at 11 significant bits or more, outputs averaged over
    # thousands of random Values
    return {"rel": 1e-3, "max": 1e-2}


# ---- inputs ----------------------------------------------------------------------------------------------------------

def _fill(cache, case, seed, lo, hi, chunk):
    """Tokens lo .. hi - 1 of every block, in chunks; the blocks of a chunk receive the same Keys and Values."""
    for i, t in enumerate(range(lo, hi, chunk)):
        n = min(chunk, hi - t)
        k, v = synth.make_kv(seed, 0, i, n, case["batch"], case["kv_heads"], t, N_OUTLIER, OUTLIER_FACTOR, device=DEVICE)
        k, v = k.contiguous(), v.contiguous()
        for layer in range(case["layers"]):
            cache.append(layer, k, v)


def _calibration_tensor(seed, stream, shape, outliers=0):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(1000003 * (seed + 1) + stream)
    x = torch.randn(shape, generator=g, device=DEVICE, dtype=torch.bfloat16)
    if outliers:
        channels = synth.outlier_channels(seed, 0, shape[2], outliers)
        gain = torch.ones(shape[2], 128)
        gain.scatter_(1, channels, OUTLIER_FACTOR)
        x *= gain.to(DEVICE, torch.bfloat16)
    return x


def prepare(case, seed):
    kind = case["kind"]
    if kind == "calibrate":
        shape = (case["tokens"], case["sequences"], case["kv_heads"], 128)
        return {"case": case, "k": _calibration_tensor(seed, 1, shape, N_OUTLIER)}
    if kind == "alpha_grid":
        shape = (case["tokens"], case["sequences"], case["kv_heads"], 128)
        q_shape = shape[:2] + (case["kv_heads"] * case["group"], 128)
        return {"case": case, "k": _calibration_tensor(seed, 1, shape, N_OUTLIER), "v": _calibration_tensor(seed, 2, shape),
                "q": _calibration_tensor(seed, 3, q_shape), "alphas": np.arange(case["alphas"]) / case["alphas"]}
    layers, batch, kv_heads, context = case["layers"], case["batch"], case["kv_heads"], case["context"]
    sample, _ = synth.make_kv(seed, 0, 0, 256, 1, kv_heads, 0, N_OUTLIER, OUTLIER_FACTOR, device=DEVICE)
    lam = np.broadcast_to(synth.make_lambda(sample).numpy(), (layers, kv_heads, 128))
    cache = Cache(layers, case["q_heads"], kv_heads, batch, case["max_tokens"], _fbits(case), lam=lam, n_sink=N_SINK,
                  window=WINDOW, evict_chunk=case["evict_chunk"], device="cuda:0")
    state = {"case": case, "cache": cache, "start": [(0, 16)] * layers, "prompt": []}
    if kind in ("decode", "layerwise"):
        _fill(cache, case, seed, 0, context, 4096)
        at = [cache.layer_state(layer) for layer in range(layers)]
        state["start"] = [(s["n_tokens"], s["cur_bits"]) for s in at]
    else:
        chunk = case.get("chunk", context)
        for i, t in enumerate(range(0, context, chunk)):
            n = min(chunk, context - t)
            blocks = [synth.make_kv(seed, layer, i, n, batch, kv_heads, t, N_OUTLIER, OUTLIER_FACTOR, device=DEVICE)
                      for layer in range(layers)]
            state["prompt"].append([(k.contiguous(), v.contiguous()) for k, v in blocks])
    # the new tokens of each step: one draw for all blocks and steps, then split up
    steps = case.get("steps", 1)
    k, v = synth.make_kv(seed, 1, 0, steps, layers * batch, kv_heads, context, 0, 1.0, device=DEVICE)
    q = torch.stack([synth.make_q(seed, 1, s, layers * batch, case["q_heads"], context + s, device=DEVICE) for s in range(steps)])
    state["k"] = list(k.view(steps, layers, batch, kv_heads, 128).contiguous())
    state["v"] = list(v.view(steps, layers, batch, kv_heads, 128).contiguous())
    state["q"] = list(q.view(steps, layers, batch, case["q_heads"], 128).contiguous())
    return state


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "calibrate":
        return calibrate_lambda(state["k"], pos_scale=case["pos_scale"])
    if kind == "alpha_grid":
        # the best alpha is the position of the smallest loss
        _, losses = alpha_grid_search(state["k"], state["q"], state["v"], case["bits"], alphas=state["alphas"],
                                      pos_scale=case["pos_scale"])
        return losses
    cache = state["cache"]
    for layer, (n, bits) in enumerate(state["start"]):
        cache.restore_layer_state(layer, n, bits)
    for blocks in state["prompt"]:
        for layer, (k, v) in enumerate(blocks):
            cache.append(layer, k, v)
    out = []
    for k, v, q in zip(state["k"], state["v"], state["q"]):
        if kind == "layerwise":
            for layer in range(case["layers"]):
                cache.append(layer, k[layer], v[layer])
                out.append(cache.decode_attention(layer, q[layer]))
        else:
            out.append(cache.decode_step(k, v, q))
    return out
