"""The one-kernel sweep of fpsa_sweep_noalloc at the edges of its layout, against the oracle's sweep.

A warp holds 2 ordinates x 16 cell chunks, a block 64 chunks, a cluster up to 8 blocks
(512 chunks), and lanes with more than 4 cells sweep them in batches: orders that do not
fill a group of ordinates, cell counts on both sides of every step, and the longest
slabs of the smallest order. The recurrence contracts (|alpha| < 1), so the rounding of a
cell (about 20 operations) and of the few map compositions does not grow along the slab:
1e-12 of the largest flux is far above it.
"""
import numpy as np
import pytest

from oracle import quadrature as qd
from oracle import transport as ot

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K", [(2, 1), (2, 65536), (4, 63), (6, 64), (10, 65), (16, 200), (16, 512), (16, 513),
                                 (34, 129), (64, 2048), (62, 2049), (128, 257), (256, 512), (254, 5)])
def test_noalloc_shapes(N, K):
    import torch
    import __graft_entry__ as g
    g.build()
    from paper_1907_13013_gb300 import binding
    rng = np.random.default_rng(N * 100000 + K)
    h = rng.uniform(0.5, 1.5, K) / K
    st = np.exp(rng.uniform(np.log(1.0), np.log(300.0), K))
    q = rng.uniform(0.0, 1.0, (K, 2, N))
    mu, _ = qd.gauss_legendre(N)
    ref = ot.sweep(mu, st, h, q)
    d = [torch.tensor(x, device="cuda:0") for x in (h, st, q)]
    psi = torch.full((K, 2, N), np.nan, dtype=torch.float64, device="cuda:0")
    binding.sweep_noalloc(N, *d, psi)
    got = psi.cpu().numpy()
    assert np.abs(got - ref).max() / np.abs(ref).max() < 1e-12
    # the flux may overwrite the source
    binding.sweep_noalloc(N, d[0], d[1], d[2], d[2])
    assert np.array_equal(d[2].cpu().numpy(), got)
