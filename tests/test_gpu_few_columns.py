"""The few-column tensor-core contractions (16, 32 or 64 columns per block, N <= 128) at
the edges of their tiles: remainders of one cell, several right-hand sides, the sizes
where the columns per block change and where the 128-column tiles take over. Each solve
is compared with the same solve on the FP32 cores: both refine the same FP64 residual to
a relative change of 1e-12 (c <= 0.99: error at most 1e-10), and the split products
(2^-16 relative) must not change the number of refinement steps by more than one.
"""
import numpy as np
import pytest

from paper_1907_13013_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,R", [(16, 9, 1), (16, 1215, 1), (16, 1217, 1), (32, 77, 3), (64, 1000, 2),
                                   (64, 4863, 1), (64, 4865, 1), (128, 8, 1), (128, 1209, 1), (128, 1217, 1),
                                   (128, 300, 5)])
def test_few_columns(N, K, R):
    import torch  # noqa: F401
    import __graft_entry__ as g
    g.build()
    from paper_1907_13013_gb300 import binding
    p = inputs.random_slab(K, N, N - 1, seed=K + N, kernel="hg", thick=(2, 60), c=(0.7, 0.99), nrhs=R)
    out = {}
    for eng in ("tensor", "simt"):
        ctx = binding.context_for(p, laplacian="wfd", precision="mixed")
        out[eng] = ctx.solve("fpsa", tol=1e-12, max_iterations=60, inner_iterations=4, contraction=eng)
        ctx.close()
    (a, sa), (b, sb) = out["tensor"], out["simt"]
    assert np.abs(a - b).max() / np.abs(b[..., 0]).max() < 1e-9
    assert abs(sa["outer_iterations"] - sb["outer_iterations"]) <= 1
