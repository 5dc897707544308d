"""One application of the tensor-core BCR solve against the dataflow solve of the same
factors: one refinement step of one inner FPSA iteration, of which all but the correction is
the same on both sides.

The split products keep about 16 bits of each factor (operand and operator in two BF16
parts, the lo x lo product left out: 2^-17 + 2^-17 + 2^-18 < 2^-15.6 a product relative to the
products of magnitudes), and so do the backward operators, which hold the couplings
multiplied in; the forward couplings keep 24 bits. A right-hand side passes one such product
in each of the 2 log2 K levels and the root, and the inverse of the FP operator is nonnegative up to small
terms, so that errors do not grow against the correction, which is no larger than the flux:
(2 levels + 1) 2^-15.6 of the largest flux bounds the difference. (BF16 alone, without the lo
parts, would err by 2^-8 a product.) Both sides' FP32 arithmetic is far below that.

The three-slice layout (2N = 384) also runs to convergence: a middle slice that pushes
nothing and couplings of 96 rows under products of 128.
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


def _both(binding, p, **kw):
    out = {}
    for eng in (2, 1):
        ctx = binding.context_for(p, laplacian="mpd", precision="mixed")
        ctx.set_tuning({"solve_engine": eng})
        assert ctx.get_tuning()["solve_engine"] == eng
        out[eng] = ctx.solve("fpsa", **kw)
        ctx.close()
    return out


@pytest.mark.parametrize("N,K,R", [(64, 200, 16), (64, 900, 40), (128, 120, 64), (192, 60, 33), (256, 40, 16)])
def test_one_application(binding, N, K, R):
    p = inputs.random_slab(K, N, N - 1, seed=2100 + K + N, kernel="hg", thick=(20, 400), c=(0.9, 0.999), nrhs=R)
    out = _both(binding, p, tol=0.0, max_iterations=1, inner_iterations=1, raise_on_notconv=False)
    a, b = out[2][0], out[1][0]
    levels = int(np.ceil(np.log2(K)))
    assert np.abs(a - b).max() / np.abs(b[..., 0]).max() < (2 * levels + 1) * 2.0 ** -15.6


@pytest.mark.parametrize("K,R", [(1, 16), (7, 16), (40, 33)])
def test_three_slices(binding, K, R):
    p = inputs.random_slab(K, 192, 191, seed=2200 + K, kernel="hg", thick=(2, 60), c=(0.7, 0.99), nrhs=R)
    out = _both(binding, p, tol=1e-12, max_iterations=60, inner_iterations=4)
    (a, sa), (b, sb) = out[2], out[1]
    assert np.abs(a - b).max() / np.abs(b[..., 0]).max() < 1e-9  # as test_gpu_bcr_paths
    assert abs(sa["outer_iterations"] - sb["outer_iterations"]) <= 1
