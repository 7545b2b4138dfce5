"""The work that users of the library have it do, as cases that can be timed and compared.

A case is one pass over a KV cache laid out ``[head][K|V][block]`` (a head here is one (layer, KV head)
stream), cut into blocks of ``n`` tokens x 128 channels.  ``kind`` says which calls the pass makes:

  prefill    eosq_encode into buffers that the program keeps, then eosq_scores of the new queries against
             the compressed keys: one step of the repository's benchmark
  roundtrip  eosq_encode, then eosq_decode of every block: an evaluation in which the cache is replaced by
             its reconstruction
  append     eosq_encode_static of the few blocks that have just filled up in one layer of a serving loop,
             then eosq_decode of them
  host       eosq_encode_host from pinned host memory and back to it
  scores     eosq_scores alone: the attention logits of one decoding step
  decode     eosq_decode alone: reading a compressed cache back

Inputs are the repository's synthetic caches (spiked model with coloured noise and outlier channels):
``recipe`` "llama" has planted ranks 2 .. 16, "ministral" ranks 1 .. 32 and 5 % pure-noise blocks, "sweep" four
spikes around the detection threshold.

What a pass returns.  The factor rows P and V carry an arbitrary common sign per factor (the method does
not define one, and the tests never compare it), and rows of P beyond a block's rank are not written.  So
the factors are compared through what a user reads out of them, the decoded blocks or the scores of the
same pass, next to the other arrays of the compressed cache.
"""
from __future__ import annotations

import math

import torch

import paper_2605_02905_b200 as eosq
from paper_2605_02905_b200 import synth

D = 128
ROTATION_SEED = 1234          # a deployment has one rotation
MEAN_RANK = 6.0               # kept factors per block, about, over these recipes
MAX_TOKENS = 1 << 24          # tokens of the largest listed cache: 16384 blocks of 1024
MAX_BLOCKS = 16384
RECIPES = {
    "llama": dict(rank_lo=2, rank_hi=16),
    "ministral": dict(rank_lo=1, rank_hi=32, noise_frac=0.05),
    "sweep": dict(fixed_theta=[5.0, 1.5, 1.05, 0.9]),
}


def _case(name, kind, heads, bph, n, bits, *, recipe="llama", dtype="f16", G=4, out="f16", full=False, keep=True):
    """heads streams of bph key and bph value blocks; ``out`` is the type that decode writes; ``full`` asks for the
    whole spectrum (the optional diagnostics); ``keep``: the program keeps its output and scratch buffers
    instead of letting the calls make new ones."""
    return dict(name=name, kind=kind, heads=heads, bph=bph, n=n, bits=bits, recipe=recipe, dtype=dtype, G=G, out=out,
                full=full, keep=keep)


def listed():
    return [
        # the smallest call there is, everything left at its default: two 256-token float32 blocks (one key, one
        # value block) of a user who tries the method out
        _case("try_out_2x256_fp32", "roundtrip", 1, 1, 256, 2, dtype="f32", out="f32", full=True, keep=False),
        # a serving loop: in one layer (8 KV heads) the next 1024 tokens are complete, 16 blocks
        _case("append_layer_16x1024", "append", 8, 1, 1024, 2),
        # prefill of one layer at 8k tokens, 128 blocks: the benchmark's one-layer shape
        _case("prefill_layer_128x1024", "prefill", 8, 8, 1024, 2),
        # prefill of the whole Llama-3.1-8B-shaped 32k cache, 16384 blocks: the benchmark's default
        _case("prefill_llama32k_16384x1024", "prefill", 256, 32, 1024, 2),
        # four layers of the Ministral-8B-shaped 64k cache at three bits, 16 queries per KV head
        _case("prefill_ministral_4096x1024_b3", "prefill", 32, 64, 1024, 3, recipe="ministral", G=16),
        # the sweep's longest blocks at four bits, whole round trip
        _case("roundtrip_sweep_512x4096_b4", "roundtrip", 8, 32, 4096, 4, recipe="sweep"),
        # the paper's own tables: square 128 x 128 blocks of a 3000-token passage, all 256 streams
        _case("roundtrip_square_11776x128", "roundtrip", 256, 23, 128, 2),
        # a ragged block length with every diagnostic array asked for, buffers made by the calls
        _case("roundtrip_ragged_304x1000_b1", "roundtrip", 8, 19, 1000, 1, out="f32", full=True, keep=False),
        # one decoding step in one layer at 32k tokens: 8 KV heads x 4 queries
        _case("scores_step_256x1024", "scores", 8, 32, 1024, 2),
        # one decoding step through eight layers at 64k tokens, batch of four: 16 queries per KV head
        _case("scores_batch_4096x1024_g16", "scores", 64, 64, 1024, 2, recipe="ministral", G=16),
        # reading half of the 32k cache back at three bits
        _case("decode_8192x1024_b3", "decode", 128, 32, 1024, 3),
        # compressing a cache that lives in host memory, four layers of the 32k cache
        _case("host_2048x1024", "host", 32, 32, 1024, 2),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["prefill", "prefill", "roundtrip", "roundtrip", "scores", "decode", "append", "host"])
    n = 8 * _log_int(rng, 16, 512)
    bits = rng.randint(1, 4)
    dtype = "f32" if kind == "roundtrip" and rng.random() < 0.25 else "f16"
    out = rng.choice(["f16", "f32"])
    blocks = MAX_BLOCKS
    tokens = MAX_TOKENS
    if kind == "append":
        blocks = eosq.eosq_encode_static_max_blocks()
    elif kind == "host":
        tokens = MAX_TOKENS // 8
    elif dtype == "f32":
        blocks = 64
    if out == "f32" or kind == "roundtrip":
        tokens //= 2
    pairs = max(1, min(blocks, tokens // n) // 2)         # (key, value) block pairs at most
    total = _log_int(rng, 1, pairs)
    heads = _log_int(rng, 1, min(256, total))
    return {k: v for k, v in _case("", kind, heads, total // heads, n, bits, recipe=rng.choice(sorted(RECIPES)), dtype=dtype,
                                   G=_log_int(rng, 1, 16), out=out, full=kind == "roundtrip" and rng.random() < 0.4,
                                   keep=rng.random() < 0.7).items() if k != "name"}


_contexts = {}


def _context():
    """The program's one context per device."""
    dev = torch.cuda.current_device()
    if dev not in _contexts:
        _contexts[dev] = eosq.Context()
    return _contexts[dev]


def prepare(case, seed):
    """Blocks (or a cache that is already compressed), queries and, where the program keeps them, output and
    scratch buffers."""
    heads, bph, n, bits, kind = case["heads"], case["bph"], case["n"], case["bits"], case["kind"]
    w = synth.kv_cache_blocks(case["recipe"], layers=1, kv_heads=heads, tokens=bph * n, n=n, device="cuda", seed=seed,
                              dtype=torch.float32 if case["dtype"] == "f32" else torch.float16, **RECIPES[case["recipe"]])
    blocks = w.blocks
    B = blocks.shape[0]
    st = dict(case=case, ctx=_context(), blocks=blocks, cache=None, workspace=None, decoded=None, scores=None)
    out_type = torch.float32 if case["out"] == "f32" else torch.float16
    if kind in ("prefill", "scores"):
        st["q"] = synth.queries(heads, case["G"], device="cuda", seed=seed + 1)
    if kind == "host":
        st["host_in"] = blocks.cpu().pin_memory()
        st["host_out"] = eosq.Cache.allocate(B, n, D, bits, pinned=True, diagnostics=False)
        st["arena"] = torch.empty(eosq.eosq_encode_host_arena_bytes(B, n, D, bits, eosq.EOSQ_F16), dtype=torch.uint8, device="cuda")
        st["blocks"] = None
        return st
    if kind in ("scores", "decode"):
        st["cache"] = eosq.Cache.allocate(B, n, D, bits, diagnostics=False)
        eosq.eosq_encode(st["ctx"], blocks, bits, ROTATION_SEED, out=st["cache"])
        st["blocks"] = None
    elif case["keep"] or kind == "append":
        st["cache"] = eosq.Cache.allocate(B, n, D, bits, diagnostics=case["full"])
        if kind != "append":
            st["workspace"] = torch.empty(eosq.eosq_workspace_bytes(B, n, D), dtype=torch.uint8, device="cuda")
    if case["keep"]:
        if kind in ("prefill", "scores"):
            st["scores"] = torch.empty((heads, case["G"], bph * n), dtype=torch.float32, device="cuda")
        else:
            st["decoded"] = torch.empty((B, n, D), dtype=out_type, device="cuda")
    return st


def _stored(cache):
    got = [cache.codes, cache.norms, cache.rank, cache.sigma, cache.phi, cache.status]
    return got + ([cache.eig, cache.lambda_plus] if cache.eig is not None else [])


def run(st):
    case, ctx = st["case"], st["ctx"]
    kind, bits, bph = case["kind"], case["bits"], case["bph"]
    out_type = torch.float32 if case["out"] == "f32" else torch.float16
    if kind == "host":
        return _stored(eosq.eosq_encode_host(ctx, st["host_in"], bits, ROTATION_SEED, st["host_out"], st["arena"]))
    if kind == "decode":
        return [eosq.eosq_decode(ctx, st["cache"], ROTATION_SEED, out_dtype=out_type, out=st["decoded"])]
    if kind == "scores":
        return [eosq.eosq_scores(ctx, st["cache"], st["q"], case["heads"], bph, 2 * bph, ROTATION_SEED, out=st["scores"])]
    if kind == "append":
        cache = eosq.eosq_encode_static(ctx, st["blocks"], bits, ROTATION_SEED, st["cache"])
    else:
        out = st["cache"]
        if out is None and not case["full"]:
            B, n, d = st["blocks"].shape
            out = eosq.Cache.allocate(B, n, d, bits, diagnostics=False)
        cache = eosq.eosq_encode(ctx, st["blocks"], bits, ROTATION_SEED, out=out, workspace=st["workspace"])
    if kind == "prefill":
        return _stored(cache) + [eosq.eosq_scores(ctx, cache, st["q"], case["heads"], bph, 2 * bph, ROTATION_SEED, out=st["scores"])]
    return _stored(cache) + [eosq.eosq_decode(ctx, cache, ROTATION_SEED, out_dtype=out_type, out=st["decoded"])]


def work(case):
    """Blocks in, compressed arrays out and in again, scores or decoded blocks out; multiply-adds of the Gram
    matrix, the eigen-decomposition (4/3 d^3), the rotation and the low-rank parts."""
    kind, n, bits, G = case["kind"], case["n"], case["bits"], case["G"]
    B = 2 * case["heads"] * case["bph"]
    stored = n * D * bits / 8 + 2 * n + 2 * MEAN_RANK * (n + D) + 136
    blocks_in = n * D * (4 if case["dtype"] == "f32" else 2)
    decoded = n * D * (4 if case["out"] == "f32" else 2)
    nbytes = flops = 0.0
    if kind in ("prefill", "roundtrip", "append", "host"):
        nbytes += B * (blocks_in + stored)
        flops += B * (4.0 * n * D * D + 4.0 / 3.0 * D ** 3 + 4.0 * n * D * MEAN_RANK)
    if kind in ("roundtrip", "append", "decode"):
        nbytes += B * (stored + decoded)
        flops += B * (2.0 * n * D * D + 2.0 * n * D * MEAN_RANK)
    if kind in ("prefill", "scores"):     # keys only
        nbytes += B / 2 * (stored + 4 * G * n) + 2 * case["heads"] * G * D
        flops += B / 2 * 2.0 * n * G * (D + MEAN_RANK)
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    """Factors and norms are stored in 16-bit floats and a residual coordinate that sits on a quantiser
    threshold may take either code.  A code's neighbour is up to 1.6 / sqrt(d) away on a unit row (one bit; less
    with more): that moves the row's decoded coordinates by up to 0.6 of the residual's root mean square and its
    score by as much, while the share of such codes is about the relative error of the rotated coordinates,
    1e-6 or less, so that the 2-norm moves by no more than 1e-3."""
    return {"rel": 1e-3, "max": 0.7, "differ": 1e-4}
