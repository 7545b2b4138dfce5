"""The exact Gram matrix on both sides of its dispatch: blocks short enough to take it at once, longer blocks that the
eigenvalue kernel queues for a second pass, and launches with few and with many blocks (the two tile shapes)."""
import numpy as np
import pytest
import torch

import oracle
import paper_2605_02905_b200 as eosq

pytestmark = pytest.mark.gpu


def _wide_spectrum_blocks(count, n, seed):
    """A strong rank-one part over weak noise: the smallest eigenvalue is below 2e-5 of the largest."""
    g = torch.Generator().manual_seed(seed)
    u, v = torch.randn(count, n, 1, generator=g), torch.randn(count, 1, 128, generator=g)
    return (u @ v + 0.05 * torch.randn(count, n, 128, generator=g)).to(torch.float16)


@pytest.mark.parametrize("n", [320, 328, 1000])
@pytest.mark.parametrize("full", [False, True])
def test_spectra_of_blocks_with_a_wide_spectrum(n, full):
    """The half-precision tensor cores would move the smallest eigenvalues here by about 1e-8 / 2e-5 = 5e-4 relative;
    from the exact Gram matrix every one agrees with the oracle's to the 1e-8 at which the iterations stop and the
    6e-8 of its storage in fp32 (held to 1e-6)."""
    ctx = eosq.Context()
    blocks = _wide_spectrum_blocks(3, n, n)
    out = eosq.Cache.allocate(3, n, 128, 2, diagnostics=True if full else "staged")
    eosq.eosq_encode(ctx, blocks.cuda(), 2, 5, out=out)
    assert eosq.eosq_check_status(ctx, out) == 0
    for b in range(3):
        sig = np.asarray(oracle.svd(blocks[b].double().numpy())[0])
        sp = oracle.eoptshrink_spectrum(n, 128, sig)
        r = sp["rank"]
        assert sig[-1] ** 2 < 1e-4 * sig[0] ** 2 and int(out.rank[b]) == r == 1
        np.testing.assert_allclose(out.sigma[b, :r].cpu().numpy(), sig[:r], rtol=1e-6)
        np.testing.assert_allclose(out.phi[b, :r].cpu().numpy(), np.asarray(sp["phi"])[:r], rtol=1e-6)
        np.testing.assert_allclose(float(out.lambda_plus[b]), sp["lambda_plus"], rtol=1e-6)
        if full:
            np.testing.assert_allclose(out.eig[b].cpu().numpy(), sig ** 2, rtol=1e-6)
    ctx.close()


@pytest.mark.parametrize("n,dtype", [(128, torch.float16), (136, torch.float32), (328, torch.float16)])
def test_few_and_many_blocks_give_the_same_bits(n, dtype):
    """300 blocks in one call against the first and the last on their own (n = 328: through the second pass)."""
    ctx = eosq.Context()
    blocks = _wide_spectrum_blocks(300, n, 7).to(dtype).cuda()
    many = eosq.eosq_encode(ctx, blocks, 3, 5)
    for b in (0, 299):
        one = eosq.eosq_encode(ctx, blocks[b:b + 1].contiguous(), 3, 5)
        for name in ("codes", "norms", "rank", "sigma", "phi", "eig"):
            assert torch.equal(getattr(one, name)[0], getattr(many, name)[b]), name
    ctx.close()


@pytest.mark.parametrize("count,launches", [(2 * 148, 8 + 2 + 1), (2 * 148 + 1, 8 + 3 + 1), (12 * 148, 8 + 3 + 1), (12 * 148 + 1, 8 + 3 + 3)])
def test_long_lists(count, launches):
    """Every block is queued.  A list of any length gives the bits of calls of one block, and a long one is reduced in the first pass's
    three launches: the band reduction of the second pass is one launch up to twelve blocks per SM only, since one costs a full list
    4 % of the call."""
    ctx = eosq.Context()
    blocks = _wide_spectrum_blocks(37, 328, 9).repeat(count // 37 + 1, 1, 1)[:count].contiguous().cuda()
    picks = (0, 36, count // 2, count - 1)
    ones = {b: eosq.eosq_encode(ctx, blocks[b:b + 1].contiguous(), 2, 5, out=eosq.Cache.allocate(1, 328, 128, 2, diagnostics="staged")) for b in picks}
    before = ctx.launch_count
    many = eosq.eosq_encode(ctx, blocks, 2, 5, out=eosq.Cache.allocate(count, 328, 128, 2, diagnostics="staged"))
    assert ctx.launch_count - before == launches
    assert eosq.eosq_check_status(ctx, many) == 0
    names = ("codes", "norms", "rank", "sigma", "phi", "V", "vr32", "coef", "lambda_plus", "status")
    for b in picks:
        for name in names:
            assert torch.equal(getattr(ones[b], name)[0], getattr(many, name)[b]), (name, b)
    first = torch.arange(count, device="cuda") % 37   # every block equals its first copy
    for name in names:
        a = getattr(many, name)
        assert torch.equal(a, a[:37][first]), name
    ctx.close()
