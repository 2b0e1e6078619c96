"""What is timed: the iterations a decoder instance runs, through the package's public entry points.

A case is one iteration of a Convertible Decoder: `rows` ongoing requests that decode one token each
and `chunks` prefill chunks of `chunk` tokens, over a paged KV cache whose pages are scattered. The
calls are Decoder.mixed_step (attention of the iteration, tensors on the device), DecoderLayer.step
(the whole decoder layer around it) and Decoder.mixed_step_host (the same step on pinned host
buffers). Sizes are those of the package's own workloads (workloads.py: config1 to config4 and the
70B-shaped trace replay), of bench.py and of the chunk-size profiler's sweep, and what lies between.

Values are N(0, 1): the softmax is then neither flat nor a single key. A step keeps the cached
lengths, so that it can be repeated; it appends its tokens to the pages all the same.
"""
import math

import numpy as np
import torch

from paper_2512_03416_b200.decoder import Decoder
from paper_2512_03416_b200.layer import DecoderLayer

TINY, SHAPE_8B, SHAPE_70B = (4, 2, 64), (32, 8, 128), (64, 8, 128)
HIDDEN, INTERMEDIATE, MAX_POSITION = 4096, 14336, 32768          # the 8B-shaped layer


def _case(kind, shape, rows, median, longest, chunks=0, chunk=0, prior=0, shortest=128, lens=2):
    """rows, median, shortest, longest: decode rows and their cached tokens (lognormal, sigma 1, clipped);
    prior: most cached tokens in front of a chunk (uniform from 0); lens: seed of those lengths."""
    return {"kind": kind, "hq": shape[0], "hkv": shape[1], "d": shape[2], "rows": rows, "median": median,
            "shortest": min(shortest, longest), "longest": longest, "chunks": chunks, "chunk": chunk, "prior": prior, "lens": lens}


def listed():
    c = [
        # the smallest iteration: a small model's mixed step, where latency and launches count
        ("tiny_mixed", _case("step", TINY, 4, 64, 128, 1, 64, shortest=16, lens=1)),
        # a decoder with hardly any load (night, or just scaled out): four requests of odd lengths
        ("decode_few_8b", _case("step", SHAPE_8B, 4, 1500, 8192, lens=7)),
        # the ordinary decode batch between bursts
        ("decode_64_8b", _case("step", SHAPE_8B, 64, 2048, 8192)),
        # a full decoder of the larger model: the replay's step without prefill work
        ("decode_203_70b", _case("step", SHAPE_70B, 203, 1200, 10240, shortest=16, lens=5)),
        # a burst: the decode batch absorbs one fresh 2048-token chunk
        ("burst_8b", _case("step", SHAPE_8B, 64, 2048, 8192, 1, 2048)),
        # long prompts in progress: chunks of 512 tokens with up to 6144 tokens before them
        ("chunked_8b", _case("step", SHAPE_8B, 128, 4096, 16384, 4, 512, prior=6144, lens=4)),
        # the replay's usual mixed step: a median prompt of odd length next to a full decode batch
        ("mixed_717_70b", _case("step", SHAPE_70B, 198, 1200, 10240, 1, 717, shortest=16, lens=6)),
        # the replay's heaviest step: the longest prompt in one chunk
        ("mixed_8192_70b", _case("step", SHAPE_70B, 190, 1200, 10240, 1, 8192, shortest=16, lens=5)),
        # an idle Convertible Decoder used as a prefiller
        ("prefill_2048_8b", _case("step", SHAPE_8B, 0, 0, 0, 1, 2048)),
        # the whole layer, at the burst and at the decode batch
        ("layer_burst_8b", _case("layer", SHAPE_8B, 64, 2048, 8192, 1, 2048)),
        ("layer_decode_8b", _case("layer", SHAPE_8B, 64, 2048, 8192)),
        # the burst end to end, from host buffers to a host buffer
        ("host_burst_8b", _case("host", SHAPE_8B, 64, 2048, 8192, 1, 2048)),
    ]
    return [dict(v, name=k) for k, v in c]


def _log(rng, lo, hi):
    """An integer from lo to hi, spread over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _cost(case):
    w = work(case)
    return max(w["bytes"] / 6.5e12, w["flops"] / 1.2e15)


def draw(rng):
    limit = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["decode", "decode", "burst", "burst", "burst", "chunked", "prefill", "tiny", "layer", "layer_decode", "host"])
        shape = rng.choice([SHAPE_8B, SHAPE_70B])
        lens, median, longest = rng.randrange(1 << 20), _log(rng, 128, 4096), rng.choice([8192, 10240, 16384])
        prior = rng.choice([0, 0, 6144])
        if kind == "decode":
            c = _case("step", shape, _log(rng, 1, 256), median, longest, shortest=16, lens=lens)
        elif kind == "burst":
            c = _case("step", shape, _log(rng, 1, 200), median, longest, 1, _log(rng, 16, 8192), prior, shortest=16, lens=lens)
        elif kind == "chunked":
            c = _case("step", shape, _log(rng, 8, 200), median, longest, rng.randint(2, 4), _log(rng, 64, 1024), 6144, shortest=16, lens=lens)
        elif kind == "prefill":
            c = _case("step", shape, 0, 0, 0, 1, _log(rng, 64, 8192), prior, lens=lens)
        elif kind == "tiny":
            c = _case("step", TINY, _log(rng, 1, 32), _log(rng, 16, 256), 512, rng.randint(0, 1), _log(rng, 2, 256), shortest=16, lens=lens)
        elif kind == "layer":
            c = _case("layer", SHAPE_8B, _log(rng, 1, 128), median, longest, 1, _log(rng, 16, 2048), prior, shortest=16, lens=lens)
        elif kind == "layer_decode":
            c = _case("layer", SHAPE_8B, _log(rng, 1, 256), median, 8192, shortest=16, lens=lens)
        else:
            c = _case("host", SHAPE_8B, _log(rng, 1, 128), median, 8192, 1, _log(rng, 64, 2048), prior, shortest=16, lens=lens)
        if _cost(c) <= limit:
            return c


def _lengths(case):
    """(cached tokens, new tokens) per row: decode rows first, then the chunks."""
    rng = np.random.default_rng(case["lens"])
    ctx = [int(min(max(round(case["median"] * math.exp(rng.standard_normal())), case["shortest"]), case["longest"]))
           for _ in range(case["rows"])]
    ctx += [int(rng.integers(0, case["prior"] + 1)) for _ in range(case["chunks"])]
    return ctx, [1] * case["rows"] + [case["chunk"]] * case["chunks"]


class _State:
    pass


def prepare(case, seed):
    ctx, q_len = _lengths(case)
    hq, hkv, d, n = case["hq"], case["hkv"], case["d"], sum(q_len)
    pages = [-(-(c + t) // 16) for c, t in zip(ctx, q_len)]
    s = _State()
    s.kind, s.ctx, s.q_len = case["kind"], ctx, q_len
    # a pool a quarter larger than the live pages, handed out in shuffled order
    s.dec = Decoder(hq, hkv, d, n_pages=-(-5 * sum(pages) // 4), max_requests=len(ctx), max_pages_per_req=max(pages), chunk_size=n,
                    alloc_shuffle_seed=seed + 1)
    gen = torch.Generator(device="cuda").manual_seed(seed)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.bfloat16)

    s.dec.pool.view(torch.bfloat16).normal_(generator=gen)                 # the cached context
    s.slots = []
    for r, (c, t) in enumerate(zip(ctx, q_len)):
        slot = s.dec.request_add(r, c + t)
        s.dec.alloc_pages(slot, c + t, for_prefill=t > 1)
        s.dec.request_set_len(slot, c)
        s.slots.append(slot)
    if s.kind == "layer":
        qd, kvd = hq * d, hkv * d

        def weight(rows, cols):
            return (normal(rows, cols) * cols ** -0.5).view(torch.int16)

        def gain():
            return (1.0 + 0.05 * normal(HIDDEN)).view(torch.int16)

        s.layer = DecoderLayer(s.dec, gain(), weight(qd + 2 * kvd, HIDDEN), weight(HIDDEN, qd), gain(), weight(INTERMEDIATE, HIDDEN),
                               weight(INTERMEDIATE, HIDDEN), weight(HIDDEN, INTERMEDIATE), max_position=MAX_POSITION)
        s.x_in = normal(n, HIDDEN).view(torch.int16)
        s.x_out = torch.empty_like(s.x_in)
        return s
    s.q, s.k_new, s.v_new = (normal(n, h, d).view(torch.int16) for h in (hq, hkv, hkv))
    s.out = torch.empty_like(s.q)
    if s.kind == "host":
        s.q, s.k_new, s.v_new, s.out = (t.cpu().pin_memory() for t in (s.q, s.k_new, s.v_new, s.out))
    return s


def run(s):
    """One iteration: its result, and the pool with the new tokens' K/V in their pages."""
    if s.kind == "layer":
        s.layer.step(s.slots, s.q_len, s.ctx, s.x_in, s.x_out, keep_len=True)
        return {"out": s.x_out.view(torch.bfloat16), "pool": s.dec.pool.view(torch.bfloat16)}
    call = s.dec.mixed_step_host if s.kind == "host" else s.dec.mixed_step
    call(s.slots, s.q_len, s.ctx, s.q, s.k_new, s.v_new, s.out, keep_len=True)
    return {"out": s.out.view(torch.bfloat16), "pool": s.dec.pool}         # the pool as it is, bit for bit


def work(case):
    """Cached K/V read once, new K/V read and written to their pages, queries (or the layer's input and
    weights) read and outputs written; flops of the visible (query, key) pairs and of the projections."""
    ctx, q_len = _lengths(case)
    hq, hkv, d, n = case["hq"], case["hkv"], case["d"], sum(q_len)
    pairs = sum(t * c + t * (t + 1) / 2 for c, t in zip(ctx, q_len))
    flops = 4.0 * d * hq * pairs
    kv = 2 * hkv * d * 2                                                    # bytes of a token's K and V
    nbytes = sum(ctx) * kv + n * kv
    if case["kind"] == "layer":
        weights = (hq + 2 * hkv) * d * HIDDEN + HIDDEN * hq * d + 3 * INTERMEDIATE * HIDDEN
        flops += 2.0 * n * weights
        nbytes += 2 * (weights + 2 * HIDDEN) + 2 * n * HIDDEN * 2
    else:
        nbytes += n * kv + 2 * n * hq * d * 2
    return {"bytes": float(nbytes), "flops": flops}


def tolerance(case):
    # About four times the difference from the same mathematics in 64 bits. Attention (bf16 inputs, weights
    # rounded to bf16 in front of the second product, bf16 result): rel 2.1e-3, max 2.4e-2. The layer (five
    # bf16 tensors in a chain, the last of which carries the input itself): rel 3.3e-3, max 1.7e-2. The
    # appended K/V of a step are copies and stay bit for bit the same.
    return {"rel": 8e-3, "max": 0.1} if case["kind"] != "layer" else {"rel": 1.3e-2, "max": 0.07}
