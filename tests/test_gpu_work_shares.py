"""How the work is dealt out, at the edges of each rule: quantiser and decode with fewer blocks than CTAs, as many, one more and
several rounds; the band reduction with two blocks per SM and one more, where its CTAs and launches change; the eigenvalue
kernel for few and for many blocks; the host path's halving chunks."""
import pytest
import torch

import paper_2605_02905_b200 as eosq
from paper_2605_02905_b200 import synth

pytestmark = pytest.mark.gpu

SMS = 148


def _blocks(count, n, seed):
    w = synth.kv_cache_blocks("llama", layers=1, kv_heads=1, tokens=n * ((count + 1) // 2), n=n, rank_hi=8, seed=seed, device="cuda")
    return w.blocks[:count].contiguous()


@pytest.mark.parametrize("n,bits", [(1000, 1), (328, 2), (1160, 3), (512, 4)])
@pytest.mark.parametrize("count", [1, SMS - 1, SMS, SMS + 1, 2 * SMS, 2 * SMS + 1, 2 * SMS + 45])
def test_every_tile_is_done_once_whoever_does_it(n, bits, count):
    """Which CTA takes a tile decides nothing about its bits: a call of `count` blocks against calls of one block (nine
    CTAs share its tiles, or fewer), into outputs that held something else before."""
    ctx = eosq.Context()
    blocks = _blocks(count, n, n + count)
    out = eosq.Cache.allocate(count, n, 128, bits, diagnostics=False)
    for name in ("codes", "norms", "P"):
        getattr(out, name).view(torch.uint8).fill_(0xA5)
    many = eosq.eosq_encode(ctx, blocks, bits, 5, out=out)
    dec = {t: eosq.eosq_decode(ctx, many, 5, out=torch.full((count, n, 128), 7.0, dtype=t, device="cuda")) for t in (torch.float16, torch.float32)}
    assert eosq.eosq_check_status(ctx, many) == 0
    for b in sorted({0, count // 2, min(count, SMS) - 1, count - 1}):
        one = eosq.eosq_encode(ctx, blocks[b:b + 1].contiguous(), bits, 5, out=eosq.Cache.allocate(1, n, 128, bits, diagnostics=False))
        r = int(one.rank[0])
        for name in ("codes", "norms", "rank"):
            assert torch.equal(getattr(one, name)[0], getattr(many, name)[b]), (name, b)
        assert torch.equal(one.P[0, :r], many.P[b, :r]) and torch.equal(one.V[0, :r], many.V[b, :r])
        for t, d in dec.items():
            assert torch.equal(eosq.eosq_decode(ctx, one, 5, out=torch.empty((1, n, 128), dtype=t, device="cuda"))[0], d[b]), (t, b)
    # the blocks in between: every norm written (none is negative, 0xA5A5 is), every row decoded
    assert bool((many.norms.view(torch.int16) >= 0).all())
    assert not any(bool((d == 7.0).all(dim=2).any()) for d in dec.values())
    ctx.close()


@pytest.mark.parametrize("count", [592, 593])
def test_eigenvalues_either_side_of_the_wide_kernel(count):
    """Both kernels stop at 1e-8 relative: singular values and shrunken ones agree with the whole spectrum's to the
    fp32 of their storage."""
    ctx = eosq.Context()
    blocks = _blocks(count, 328, 3)
    out = eosq.eosq_encode(ctx, blocks, 2, 5, out=eosq.Cache.allocate(count, 328, 128, 2, diagnostics="staged"))
    full = eosq.eosq_encode(ctx, blocks, 2, 5, out=eosq.Cache.allocate(count, 328, 128, 2, diagnostics=True))
    assert eosq.eosq_check_status(ctx, out) == 0 and torch.equal(out.rank, full.rank)
    kept = torch.arange(out.sigma.shape[1], device="cuda")[None, :] < out.rank[:, None]
    for name in ("sigma", "phi"):
        a, b = getattr(out, name)[kept], getattr(full, name)[kept]
        assert float(((a - b).abs() / b.abs()).max()) < 1e-6, name
    ctx.close()


@pytest.mark.parametrize("count,n", [(1, 4096), (300, 1000), (600, 1024)])
def test_host_chunks_that_halve(count, n):
    """One chunk; 150, 75 and 75 blocks; 300, 150, 75 and 75."""
    ctx = eosq.Context()
    blocks = _blocks(count, n, 11)
    dev = eosq.eosq_encode(ctx, blocks, 2, 5, out=eosq.Cache.allocate(count, n, 128, 2, diagnostics=False))
    out = eosq.Cache.allocate(count, n, 128, 2, pinned=True, diagnostics=False)
    arena = torch.empty(eosq.eosq_encode_host_arena_bytes(count, n, 128, 2, eosq.EOSQ_F16), dtype=torch.uint8, device="cuda")
    eosq.eosq_encode_host(ctx, blocks.cpu().pin_memory(), 2, 5, out, arena)
    torch.cuda.synchronize()
    for name in ("codes", "norms", "rank", "status"):
        assert torch.equal(getattr(out, name), getattr(dev, name).cpu()), name
    ctx.close()


@pytest.mark.parametrize("n,count,chunks", [(1024, 64, 1), (1024, 65, 1), (1024, 95, 1), (1024, 96, 2), (1024, 128, 2), (4096, 17, 1), (4096, 24, 2),
                                            (4096, 47, 2), (4096, 48, 3)])
def test_host_chunks_leave_no_crumbs(n, count, chunks):
    """Every chunk pays a whole chain of launches: a rest of less than one and a half times 16 MiB is one chunk."""
    ctx = eosq.Context()
    blocks = _blocks(count, n, 12)
    eosq.eosq_encode(ctx, blocks[:1].contiguous(), 2, 5)
    chain = ctx.launch_count
    out = eosq.Cache.allocate(count, n, 128, 2, pinned=True, diagnostics=False)
    arena = torch.empty(eosq.eosq_encode_host_arena_bytes(count, n, 128, 2, eosq.EOSQ_F16), dtype=torch.uint8, device="cuda")
    eosq.eosq_encode_host(ctx, blocks.cpu().pin_memory(), 2, 5, out, arena)
    assert ctx.launch_count == chain * (1 + chunks)
    ctx.close()


@pytest.mark.parametrize("n", [328, 256])
def test_chasing_either_side_of_its_line(n):
    """1776 blocks are chased by two warps per pair of matrices, 1777 by one, and an odd last matrix keeps itself company: the same
    bits (n = 256: from the exact Gram matrix)."""
    ctx = eosq.Context()
    blocks = _blocks(12 * SMS + 1, n, 21)
    whole = eosq.eosq_encode(ctx, blocks, 2, 5, out=eosq.Cache.allocate(12 * SMS + 1, n, 128, 2, diagnostics="staged"))
    assert eosq.eosq_check_status(ctx, whole) == 0
    for count in (12 * SMS, SMS + 1, SMS, 7, 1):
        part = eosq.eosq_encode(ctx, blocks[:count].contiguous(), 2, 5, out=eosq.Cache.allocate(count, n, 128, 2, diagnostics="staged"))
        for name in ("codes", "norms", "rank", "sigma", "phi", "V", "vr32", "coef", "lambda_plus", "status"):
            assert torch.equal(getattr(part, name), getattr(whole, name)[:count]), (name, count)
    ctx.close()


@pytest.mark.parametrize("n", [328, 128])
def test_kept_vectors_either_side_of_their_line(n):
    """2960 blocks have their vectors back-transformed with one barrier per stage, 2961 with two: the same bits."""
    ctx = eosq.Context()
    blocks = _blocks(20 * SMS + 1, n, 22)
    whole = eosq.eosq_encode(ctx, blocks, 2, 5, out=eosq.Cache.allocate(20 * SMS + 1, n, 128, 2, diagnostics="staged"))
    assert eosq.eosq_check_status(ctx, whole) == 0
    part = eosq.eosq_encode(ctx, blocks[:-1].contiguous(), 2, 5, out=eosq.Cache.allocate(20 * SMS, n, 128, 2, diagnostics="staged"))
    for name in ("rank", "sigma", "phi", "V", "vr32", "coef", "lambda_plus", "status", "codes"):
        assert torch.equal(getattr(part, name), getattr(whole, name)[:-1]), name
    ctx.close()
