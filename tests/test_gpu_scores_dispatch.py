"""The score kernel on both sides of its dispatch: 8 and 16 queries per pass and more than one pass, heads whose W = Pi q the
CTAs make themselves and heads whose W a kernel in front makes, and block lengths whose last stage of four tiles holds one."""
import math

import pytest
import torch

import paper_2605_02905_b200 as eosq
from paper_2605_02905_b200 import synth

import parity

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,bits,G,heads,bph", [
    (128, 2, 4, 40, 9),     # one tile per block: every stage holds a lone tile
    (520, 3, 16, 3, 5),     # five tiles, the last one lone and ragged
    (136, 4, 9, 300, 1),    # more heads than CTAs: W from the kernel in front
    (136, 2, 16, 300, 1),   # the same with an order of coordinates of its own; a CTA's third head
    (264, 2, 12, 301, 1),   # and a last working CTA with one block where the others have three
    (136, 3, 8, 301, 1),
    (640, 1, 33, 2, 3),     # three passes
    (256, 2, 8, 149, 2),    # two CTAs share a head, some touch two
])
def test_scores_at_the_edges_of_the_dispatch(n, bits, G, heads, bph):
    ctx = eosq.Context()
    w = synth.kv_cache_blocks("scores", layers=1, kv_heads=heads, tokens=bph * n, n=n, rank_hi=8, seed=n, device="cuda")
    cache = eosq.eosq_encode(ctx, w.blocks, bits, 7, out=eosq.Cache.allocate(2 * heads * bph, n, 128, bits, diagnostics=False))
    q = synth.queries(heads, G, seed=2).cuda()
    s = eosq.eosq_scores(ctx, cache, q, heads, bph, 2 * bph, 7)
    assert eosq.eosq_check_status(ctx, cache) == 0
    pairs = [(0, 0), (0, bph - 1), (heads // 2, bph // 2), (heads - 1, bph - 1)]
    parity.compare_scores(cache, q, s, heads, bph, 2 * bph, bits, 7, 1.0 / math.sqrt(128), pairs=pairs)
    # every block once more against the decoded keys in fp32: 1e-3 of the score's own scale, as in the comparison above
    keys = eosq.eosq_decode(ctx, cache, 7).view(heads, 2, bph * n, 128)[:, 0]
    want = torch.einsum("hgd,htd->hgt", q.float(), keys) / math.sqrt(128)
    scale = want.abs() + q.float().norm(dim=2)[:, :, None] * keys.norm(dim=2)[:, None, :] / 128
    assert float(((s - want).abs() / scale).max()) < 1e-3
    ctx.close()


def test_negative_rank_words_count_as_zero():
    """In a cache written elsewhere: no factor rows are announced to a stage's barrier, and none are added (decode likewise)."""
    ctx = eosq.Context()
    w = synth.kv_cache_blocks("scores", layers=1, kv_heads=2, tokens=2 * 520, n=520, rank_hi=8, seed=1, device="cuda")
    cache = eosq.eosq_encode(ctx, w.blocks, 2, 7, out=eosq.Cache.allocate(8, 520, 128, 2, diagnostics=False))
    q = synth.queries(2, 4, seed=2).cuda()
    got = {}
    for word in (0, -1, -5, -2**31):
        cache.rank.fill_(word)
        got[word] = eosq.eosq_scores(ctx, cache, q, 2, 2, 4, 7), eosq.eosq_decode(ctx, cache, 7)
        assert eosq.eosq_check_status(ctx, cache) == 0
        assert all(torch.equal(a, b) for a, b in zip(got[word], got[0])), word
    ctx.close()


@pytest.mark.parametrize("n,bits,G", [(264, 2, 4), (392, 2, 16), (648, 2, 9), (896, 1, 4), (1160, 2, 16), (1544, 4, 8), (392, 3, 4), (1160, 3, 16)])
def test_scores_whichever_group_takes_a_tile(n, bits, G):
    """Three groups take turns on the tiles, four of which make a stage: 3, 4, 6, 7, 10 and 13 tiles per block shift the groups' turns
    from block to block, and leave groups without a tile in a block's last stage.  Against the decoded keys, to 1e-3 of the
    score's own scale; every block of a CTA's run takes part."""
    ctx = eosq.Context()
    heads, bph = 2, 150   # three blocks each for a hundred CTAs
    w = synth.kv_cache_blocks("scores", layers=1, kv_heads=heads, tokens=bph * n, n=n, rank_hi=11, seed=n, device="cuda")
    cache = eosq.eosq_encode(ctx, w.blocks, bits, 7, out=eosq.Cache.allocate(2 * heads * bph, n, 128, bits, diagnostics=False))
    q = synth.queries(heads, G, seed=2).cuda()
    s = eosq.eosq_scores(ctx, cache, q, heads, bph, 2 * bph, 7, out=torch.full((heads, G, bph * n), float("nan"), device="cuda"))
    assert eosq.eosq_check_status(ctx, cache) == 0
    keys = eosq.eosq_decode(ctx, cache, 7).view(heads, 2, bph * n, 128)[:, 0]
    want = torch.einsum("hgd,htd->hgt", q.double(), keys.double()) / math.sqrt(128)
    scale = want.abs() + q.double().norm(dim=2)[:, :, None] * keys.double().norm(dim=2)[:, None, :] / 128
    assert float(((s - want).abs() / scale).max()) < 1e-3
    ctx.close()


@pytest.mark.parametrize("G", [4, 16])
def test_error_of_the_sums_against_64_bits(G):
    """Scores from what the cache stores, in 64 bits, next to the library's.  With one-bit codes, whose centroids the operands hold
    exactly, what is left is the operands' split into two halves (2^-22) and the sums in fp32: an error of 1.18e-7 of the scores while
    none of those runs over more than sixteen products side by side (per seed 1.15 to 1.27e-7), 1.33e-7 with sixteen queries (1.30 to
    1.36e-7) when they ran over 32.  The line lies half-way, for the mean of six."""
    ctx, heads, bph, seed = eosq.Context(), 4, 12, 1234
    pi = torch.tensor(eosq.eosq_rotation(128, seed), device="cuda")
    cen = torch.tensor(eosq.eosq_codebook(1, 128)[0], device="cuda")
    got = []
    for n in (136, 1024):
        for draw in (1, 2, 3):
            w = synth.kv_cache_blocks("llama", layers=1, kv_heads=heads, tokens=bph * n, n=n, seed=draw, device="cuda")
            B = w.blocks.shape[0]
            c = eosq.eosq_encode(ctx, w.blocks, 1, seed, out=eosq.Cache.allocate(B, n, 128, 1, diagnostics=False))
            q = synth.queries(heads, G, device="cuda", seed=draw + 1)
            s = eosq.eosq_scores(ctx, c, q, heads, bph, 2 * bph, seed)
            assert eosq.eosq_check_status(ctx, c) == 0
            idx = ((c.codes.view(B, n, 16, 1).long() >> torch.arange(8, device="cuda")) & 1).view(B, n, 128)
            kept = (torch.arange(eosq.EOSQ_RMAX, device="cuda")[None] < c.rank[:, None])[:, :, None]
            P, V = (torch.where(kept, a.view(torch.float16).double().view(B, eosq.EOSQ_RMAX, -1), 0.0) for a in (c.P, c.V))
            x = torch.einsum("bit,bij->btj", P, V) + c.norms.view(torch.float16).double().view(B, n, 1) * (cen[idx] @ pi)
            want = torch.einsum("hgd,htd->hgt", q.double(), x.view(heads, 2, bph * n, 128)[:, 0]) / math.sqrt(128)
            got.append(float((s.double() - want).norm() / want.norm()))
    assert sum(got) / len(got) < 1.25e-7, got
    ctx.close()
