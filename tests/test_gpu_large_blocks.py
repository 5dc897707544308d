"""Factorizations whose blocks are inverted outside the register-tiled kernels: the level
kernels k_bcr_schur (one register tile per order range), k_bamax and k_btranspose at the
edges of their tiles, through the solution.

The FP correction only preconditions, so a wrong factor shows as a changed iteration
count or a failure to converge: the iteration counts must match the oracle's within one
(the correction's rounding, FP64 both) and the converged flux its direct solution. Both
sides iterate to 1e-12, so errors in the flux are at most 1e-12 c / (1 - c) < 1e-9.
"""
import numpy as np
import pytest

from oracle import iterations as oit
from paper_1907_13013_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,precision", [(2, 9, "fp64"), (8, 21, "fp64"), (128, 5, "fp64"), (128, 14, "mixed"),
                                           (160, 7, "fp64"), (256, 5, "mixed"), (256, 6, "fp64")])
def test_level_kernels(N, K, precision):
    import torch  # noqa: F401
    import __graft_entry__ as g
    g.build()
    from paper_1907_13013_gb300 import binding
    p = inputs.random_slab(K, N, N - 1, seed=900 + N, kernel="hg", thick=(2, 60), c=(0.8, 0.99))
    ctx = binding.context_for(p, laplacian="mpd", precision=precision)
    phi, st = ctx.solve("fpsa", tol=1e-12, max_iterations=300)
    ctx.close()
    ref = oit.direct_solve(p)
    assert np.abs(phi[0] - ref).max() / np.abs(ref[..., 0]).max() < 1e-9
    if precision == "fp64":
        _, n = oit.fpsa_source_iteration(p, "mpd", tol=1e-12, max_it=300)
        assert abs(st["iterations"] - n) <= 1
