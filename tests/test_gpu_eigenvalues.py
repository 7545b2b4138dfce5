"""Eigenvalues and kept vectors where they are hardest to tell apart: pairs of kept singular values whose eigenvalues are
close, and the kernels that a block's eigenvalues may come from."""
import numpy as np
import pytest
import torch

import oracle
import paper_2605_02905_b200 as eosq
from paper_2605_02905_b200 import synth

pytestmark = pytest.mark.gpu

N, D, PER_GAP = 160, 128, 16
GAPS = (1e-5, 1e-6, 3e-7, 1e-7, 5e-8, 2e-8)


def _close_pair_blocks(seed):
    """fp32 blocks with five strong singular values, two of which have eigenvalues that differ by `gap` relative.  Storing
    a block in fp32 moves a strong singular value by some 6e-8 / sqrt(N D) of itself, which is far less than the smallest gap."""
    rng = np.random.default_rng(seed)
    blocks, gaps = [], []
    for gap in GAPS:
        for _ in range(PER_GAP):
            u, _ = np.linalg.qr(rng.standard_normal((N, D)))
            v, _ = np.linalg.qr(rng.standard_normal((D, D)))
            s = np.concatenate([[40.0, 30.0, 25.0, 20.0, 10.0], rng.uniform(0.8, 1.2, D - 5)])
            lower = rng.integers(0, 4)
            s[lower + 1] = s[lower] * np.sqrt(1.0 - gap)
            blocks.append((u * s) @ v.T)
            gaps.append(gap)
    return torch.tensor(np.stack(blocks), dtype=torch.float32), np.array(gaps)


@pytest.mark.parametrize("count,diagnostics", [(len(GAPS) * PER_GAP, "staged"), (600, "staged"), (len(GAPS) * PER_GAP, True)])
def test_kept_vectors_of_close_pairs_are_orthogonal(count, diagnostics):
    """A kept vector comes from its computed eigenvalue by one solve, so an eigenvalue that is off by delta leaves
    delta / gap of its neighbour in it.  The eigenvalues are good to 1e-14 relative (rounding of the reduction,
    some sqrt(128) 1e-16, and the iterations' end), twice that per pair; the vectors are stored in fp32 (6e-8)."""
    ctx = eosq.Context()
    blocks, gaps = _close_pair_blocks(3)
    unique = len(blocks)
    dev = blocks.cuda().repeat((count + unique - 1) // unique, 1, 1)[:count].contiguous()
    out = eosq.eosq_encode(ctx, dev, 2, 5, out=eosq.Cache.allocate(count, N, D, 2, diagnostics=diagnostics))
    assert eosq.eosq_check_status(ctx, out) == 0
    assert bool((out.rank == 5).all())
    v = out.vr32[:, :5].double()
    off = (v @ v.transpose(1, 2) - torch.eye(5, dtype=torch.float64, device="cuda")).abs().amax(dim=(1, 2)).cpu().numpy()
    bound = 5e-7 + 2e-14 / np.resize(gaps, count)
    worst = {g: float(off[np.resize(gaps, count) == g].max()) for g in GAPS}
    assert (off <= bound).all(), worst
    ctx.close()


@pytest.mark.parametrize("n,diagnostics", [(1000, "staged"), (1000, True), (256, "staged")])
def test_bits_do_not_depend_on_the_number_of_blocks(n, diagnostics):
    """600 blocks in one call, which takes the kernel with a warp per block unless the whole spectrum is asked for, against the
    same blocks in calls of 300 and of one, which take a CTA per block.  Planted ranks up to 16: ranks 10 and 11
    read two more eigenvalues."""
    ctx = eosq.Context()
    count = 600
    w = synth.kv_cache_blocks("many", layers=1, kv_heads=4, tokens=75 * n, n=n, rank_lo=6, rank_hi=16, seed=n, device="cuda")
    blocks = w.blocks[:count].contiguous()
    many = eosq.eosq_encode(ctx, blocks, 2, 5, out=eosq.Cache.allocate(count, n, D, 2, diagnostics=diagnostics))
    assert int((many.rank >= 10).sum()) > 0 and int((many.rank < 10).sum()) > 0
    kept = torch.arange(eosq.EOSQ_RMAX, device="cuda")[None, :] < many.rank[:, None]
    for first, size in ((0, 300), (300, 300), (0, 1), (599, 1)):
        part = slice(first, first + size)
        few = eosq.eosq_encode(ctx, blocks[part].contiguous(), 2, 5, out=eosq.Cache.allocate(size, n, D, 2, diagnostics="staged"))
        for name in ("codes", "norms", "rank", "sigma", "phi", "V", "status", "lambda_plus", "vr32", "coef"):
            assert torch.equal(getattr(few, name), getattr(many, name)[part]), (name, first, size)
        assert torch.equal(few.P[kept[part]], many.P[part][kept[part]])
    ctx.close()


def test_blocks_without_a_finite_entry_are_flagged():
    """Whichever kernel runs: a Gram matrix that is NaN all over has no finite entry to scale by, and is not a zero matrix."""
    ctx = eosq.Context()
    blocks = torch.zeros(600, 328, D, dtype=torch.float16, device="cuda")
    blocks[1::2] = float("nan")
    for count, diagnostics in ((2, False), (600, False), (2, True)):
        out = eosq.eosq_encode(ctx, blocks[:count].contiguous(), 2, 5, out=eosq.Cache.allocate(count, 328, D, 2, diagnostics=diagnostics))
        assert bool((out.status[0::2] == 0).all()) and bool((out.status[1::2] != 0).all()), (count, diagnostics)
    ctx.close()


@pytest.mark.parametrize("channels", [48, 64, 100])
@pytest.mark.parametrize("front", [True, False])
def test_spectra_of_singular_blocks(channels, front):
    """Blocks with channels that are zero throughout: rows of the reduced matrix that are zero, or rounding of the rest, where the
    counts' recurrences meet their smallest factors.  The eigenvalues that are not zero to the fp32 of their storage and the 1e-8 at which
    the iterations stop (1e-6, as in the other tests), the zeros to the 2e-15 at which brackets end and the rounding of the reduction,
    some 128 of 1e-16 of the largest (2e-14 in all); no block flagged, and the kept values those of the oracle."""
    ctx = eosq.Context()
    rng = np.random.default_rng(channels)
    blocks = np.zeros((6, N, D), dtype=np.float32)
    for b in range(6):
        where = np.arange(channels) if front else np.sort(rng.permutation(D)[:channels])
        noise = rng.standard_normal((N, channels))
        for s in (8.0, 5.0):
            noise += s * np.outer(rng.standard_normal(N), rng.standard_normal(channels)) / np.sqrt(channels)
        blocks[b][:, where] = noise
    full = eosq.eosq_encode(ctx, torch.tensor(blocks, device="cuda"), 2, 5)
    few = eosq.eosq_encode(ctx, torch.tensor(blocks, device="cuda"), 2, 5, out=eosq.Cache.allocate(6, N, D, 2, diagnostics="staged"))
    assert eosq.eosq_check_status(ctx, full) == 0 and eosq.eosq_check_status(ctx, few) == 0
    for b in range(6):
        sig = np.asarray(oracle.svd(blocks[b].astype(np.float64))[0])
        eig = full.eig[b].cpu().numpy()
        np.testing.assert_allclose(eig[:channels], sig[:channels] ** 2, rtol=1e-6)
        assert np.abs(eig[channels:]).max() < 2e-14 * sig[0] ** 2
        sp = oracle.eoptshrink_spectrum(N, D, sig)
        r = sp["rank"]
        for out in (full, few):
            assert int(out.rank[b]) == r > 0
            np.testing.assert_allclose(out.sigma[b, :r].cpu().numpy(), sig[:r], rtol=1e-6)
            np.testing.assert_allclose(out.phi[b, :r].cpu().numpy(), np.asarray(sp["phi"])[:r], rtol=1e-6)
    ctx.close()
