"""The segmented sweep's default chunk length on many short slabs: no longer than gives each
of a block's eight warps a chunk of the longest slab (a longer one leaves warps without
cells), and the sweeps are right there, slab by slab, against the oracle's direct solution
(converged to 1e-12 with c <= 0.9: errors below 1e-10).
"""
import numpy as np
import pytest

from oracle import iterations as oit
from paper_1907_13013_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_many_short_slabs(precision):
    import torch  # noqa: F401
    import __graft_entry__ as g
    g.build()
    from paper_1907_13013_gb300 import binding
    kinds = [inputs.random_slab(K, 16, 15, seed=1900 + K, kernel="hg", thick=(2, 20), c=(0.5, 0.9))
             for K in (40, 17, 1, 33)]
    slabs = [kinds[b % 4] for b in range(6000)]
    ctx = binding.context_for(slabs, laplacian="mpd", precision=precision)
    assert ctx.get_tuning()["sweep_cells_per_thread"] <= 5
    phi, _ = ctx.solve("fpsa", tol=1e-12, max_iterations=300)
    ctx.close()
    ref = np.concatenate([oit.direct_solve(p) for p in kinds])
    got = phi[0].reshape((1500,) + ref.shape)
    assert np.abs(got - ref).max() / np.abs(ref[..., 0]).max() < 1e-9
