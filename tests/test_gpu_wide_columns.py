"""The contractions of orders above 128 at the edges of their column tiles, against SIMT.

Tiles hold 64 columns (32 cells): one cell, a tile less or more one cell, several
right-hand sides (a tile never spans two), orders whose second row tile is partly empty,
and GMRES (the single-GEMM kinds). The operators are split with a relative error of 2^-16,
which only the inner (preconditioning) iterations see: both engines converge to 1e-12 with
c <= 0.99, so the fluxes agree to 1e-9, and FPSA's refinement steps differ by at most one.
"""
import numpy as np
import pytest

from paper_1907_13013_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    import __graft_entry__ as g
    g.build()
    from paper_1907_13013_gb300 import binding as b
    return b


@pytest.mark.parametrize("method", ["fpsa", "gmres"])
@pytest.mark.parametrize("N,K,R", [(160, 1, 1), (192, 31, 2), (224, 33, 1), (256, 32, 3)])
def test_wide_columns(binding, N, K, R, method):
    p = inputs.random_slab(K, N, N - 1, seed=1100 + K + N, kernel="hg", thick=(2, 60), c=(0.7, 0.99), nrhs=R)
    out = {}
    for eng in ("tensor", "simt"):
        ctx = binding.context_for(p, laplacian="mpd", precision="mixed")
        out[eng] = ctx.solve(method, tol=1e-12, max_iterations=100, inner_iterations=4 if method == "fpsa" else 0,
                             contraction=eng)
        ctx.close()
    (a, sa), (b, sb) = out["tensor"], out["simt"]
    assert np.abs(a - b).max() / np.abs(b[..., 0]).max() < 1e-9
    assert method == "gmres" or abs(sa["outer_iterations"] - sb["outer_iterations"]) <= 1
