"""Orders whose blocks are halved twice to an odd size by the recursive inversion (2N = 4 x odd
above what one CTA inverts after one halving): the leaves' shared memory is sized for the odd
order. As test_gpu_large_blocks: FP64 iteration counts within one of the oracle's, and the
flux of its direct solution (both sides to 1e-12, c <= 0.99: 1e-9)."""
import numpy as np
import pytest

from oracle import iterations as oit
from paper_1907_13013_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,precision", [(170, 3, "fp64"), (194, 4, "fp64"), (254, 3, "fp64"), (242, 4, "mixed"),
                                           (254, 3, "mixed")])
def test_odd_leaves(N, K, precision):
    import torch  # noqa: F401
    import __graft_entry__ as g
    g.build()
    from paper_1907_13013_gb300 import binding
    p = inputs.random_slab(K, N, N - 1, seed=2500 + N, kernel="hg", thick=(2, 60), c=(0.8, 0.99))
    ctx = binding.context_for(p, laplacian="mpd", precision=precision)
    phi, st = ctx.solve("fpsa", tol=1e-12, max_iterations=300)
    ctx.close()
    ref = oit.direct_solve(p)
    assert np.abs(phi[0] - ref).max() / np.abs(ref[..., 0]).max() < 1e-9
    if precision == "fp64":
        _, n = oit.fpsa_source_iteration(p, "mpd", tol=1e-12, max_it=300)
        assert abs(st["iterations"] - n) <= 1
