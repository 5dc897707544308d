"""The Schur update kernel at the edges of its register tiles (1 to 8 outputs of 16 rows and
columns a thread), through the solution, as test_gpu_large_blocks: the correction only
preconditions, so a wrong update shows as a changed iteration count or a failure to
converge. FP64 counts must match the oracle's within one; both sides iterate to 1e-12 with
c <= 0.99, so fluxes agree to 1e-9.
"""
import numpy as np
import pytest

from oracle import iterations as oit
from paper_1907_13013_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K", [(4, 33), (6, 18), (14, 9), (18, 12), (34, 8), (40, 11), (62, 5), (66, 7), (94, 5),
                                 (98, 6), (130, 6), (162, 5), (194, 4), (226, 3)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_tiles(N, K, precision):
    import torch  # noqa: F401
    import __graft_entry__ as g
    g.build()
    from paper_1907_13013_gb300 import binding
    p = inputs.random_slab(K, N, N - 1, seed=2300 + N, kernel="hg", thick=(2, 60), c=(0.8, 0.99))
    ctx = binding.context_for(p, laplacian="mpd", precision=precision)
    phi, st = ctx.solve("fpsa", tol=1e-12, max_iterations=300)
    ctx.close()
    ref = oit.direct_solve(p)
    assert np.abs(phi[0] - ref).max() / np.abs(ref[..., 0]).max() < 1e-9
    if precision == "fp64":
        _, n = oit.fpsa_source_iteration(p, "mpd", tol=1e-12, max_it=300)
        assert abs(st["iterations"] - n) <= 1
