"""The BCR solves at the edges of their layouts, through converged solutions.

test_packets: the dataflow solve (staged and unstaged blocks, 1 to 8 right-hand sides per
unit, with and without a coarse step, one and two blocks per SM, FP64's two-word packets).
Its sums run in a fixed order, so repeated solves give the same bits; the flux is compared
with the oracle's direct solution: both sides iterate to 1e-12 with c <= 0.99, so errors are
below 1e-10.

test_tensor_core: the tensor-core solve (1, 2 and 4 row slices per cell, ragged tiles of
right-hand sides, one cell, levels with and without right neighbours) against the dataflow
solve of the same factors. The correction only preconditions: split products (2^-16
relative) must not change the refinement steps by more than one, and both converge to the
same flux.
"""
import numpy as np
import pytest

from oracle import iterations as oit
from paper_1907_13013_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    import __graft_entry__ as g
    g.build()
    from paper_1907_13013_gb300 import binding as b
    return b


@pytest.mark.parametrize("N,K,R,precision", [(16, 1, 1, "fp64"), (16, 2, 1, "mixed"), (16, 200, 1, "fp64"),
                                             (16, 1300, 1, "mixed"), (32, 37, 3, "mixed"), (64, 300, 8, "mixed"),
                                             (64, 33, 2, "fp64"), (128, 60, 5, "mixed"), (8, 19, 9, "fp64")])
def test_packets(binding, N, K, R, precision):
    p = inputs.random_slab(K, N, N - 1, seed=500 + K + N, kernel="hg", thick=(2, 60), c=(0.7, 0.99), nrhs=R)
    ctx = binding.context_for(p, laplacian="wfd", precision=precision)
    phi, _ = ctx.solve("fpsa", tol=1e-12, max_iterations=300)
    again, _ = ctx.solve("fpsa", tol=1e-12, max_iterations=300)
    ctx.close()
    assert np.array_equal(phi, again)
    for r in {0, R - 1}:
        ref = oit.direct_solve(dict(p, Q=p["Q"][r]))
        assert np.abs(phi[r] - ref).max() / np.abs(ref[..., 0]).max() < 1e-9


@pytest.mark.parametrize("N,K,R", [(64, 1, 16), (64, 2, 17), (64, 75, 33), (64, 130, 64), (128, 3, 65), (128, 40, 48),
                                   (256, 5, 16), (256, 12, 64)])
def test_tensor_core(binding, N, K, R):
    p = inputs.random_slab(K, N, N - 1, seed=700 + K + N, kernel="hg", thick=(2, 60), c=(0.7, 0.99), nrhs=R)
    out = {}
    for eng in (2, 1):
        ctx = binding.context_for(p, laplacian="mpd", precision="mixed")
        ctx.set_tuning({"solve_engine": eng})
        assert ctx.get_tuning()["solve_engine"] == eng
        out[eng] = ctx.solve("fpsa", tol=1e-12, max_iterations=60, inner_iterations=4)  # step for step
        ctx.close()
    (a, sa), (b, sb) = out[2], out[1]
    assert np.abs(a - b).max() / np.abs(b[..., 0]).max() < 1e-9
    assert abs(sa["outer_iterations"] - sb["outer_iterations"]) <= 1
