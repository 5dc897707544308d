"""The dataflow BCR solve with 2 to 15 right-hand sides, in units of 2, 4 and 8 that read
several elements a thread at a time, against the same solve of each right-hand side alone:
one refinement step of one inner FPSA iteration (FP64: one iteration), of which only the
correction depends on the units. Both sides sum at most 2N products in each of 2 log2 K + 1
levels, in different orders: (2 levels + 1) 2N units of rounding of the largest flux bound
the difference. Orders of staged and unstaged blocks, remainders of every unit size, levels
with and without right neighbours, and repeated solves equal to the bit.
"""
import numpy as np
import pytest

from paper_1907_13013_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,eps", [("mixed", 2.0 ** -24), ("fp64", 2.0 ** -53)])
@pytest.mark.parametrize("N,K,R", [(8, 33, 3), (16, 40, 9), (30, 21, 5), (32, 100, 3), (64, 70, 8), (64, 19, 2), (80, 37, 13),
                                   (128, 24, 4), (128, 33, 8), (160, 11, 7), (256, 9, 3), (250, 6, 15)])
def test_chunks(precision, eps, N, K, R):
    import torch  # noqa: F401
    import __graft_entry__ as g
    g.build()
    from paper_1907_13013_gb300 import binding
    p = inputs.random_slab(K, N, N - 1, seed=2400 + K + N, kernel="hg", thick=(20, 400), c=(0.9, 0.999), nrhs=R)
    kw = dict(tol=0.0, max_iterations=1, inner_iterations=1, raise_on_notconv=False)

    def solve(q):
        ctx = binding.context_for(q, laplacian="mpd", precision=precision)
        assert ctx.get_tuning()["solve_engine"] == 1
        phi, _ = ctx.solve("fpsa", **kw)
        again, _ = ctx.solve("fpsa", **kw)
        ctx.close()
        assert np.array_equal(phi, again)
        return phi
    together = solve(p)
    levels = int(np.ceil(np.log2(K)))
    for r in range(R):
        alone = solve(dict(p, Q=p["Q"][r:r + 1]))
        assert np.abs(together[r] - alone[0]).max() / np.abs(alone[..., 0]).max() < (2 * levels + 1) * 2 * N * eps
