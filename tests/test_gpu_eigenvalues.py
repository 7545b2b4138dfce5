"""Eigenvalues and kept vectors where they are hardest to tell apart: pairs of kept singular values whose eigenvalues are
close, with the largest eigenvalues only and with the whole spectrum."""
import numpy as np
import pytest
import torch

import paper_2605_02905_b200 as eosq

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


@pytest.mark.parametrize("count,diagnostics", [(len(GAPS) * PER_GAP, "staged"), (len(GAPS) * PER_GAP, True)])
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
