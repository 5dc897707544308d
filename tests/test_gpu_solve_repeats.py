"""Repeated solves of one context give the same bits: the BCR solves sum in an order that
does not depend on timing. With a fixed number of inner iterations nothing else in a solve
does either (integer maxima, fixed dot trees), so every difference would be a value read or
written out of turn.

test_coarse_step: the staged dataflow solve with its coarse step, at the orders whose copy
ring has three stages (an odd number: a stage passes from one compute group of a block to
the other) and at one with four.
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


def _repeat(binding, p, times, method, precision, **kw):
    ctx = binding.context_for(p, laplacian="wfd", precision=precision)
    kw["tol"] = 1e-12 if method == "fpsa" else 1e-10
    first, s0 = ctx.solve(method, max_iterations=300, **kw)
    for _ in range(times - 1):
        again, s1 = ctx.solve(method, max_iterations=300, **kw)
        assert np.array_equal(first, again)
        assert s1["iterations"] == s0["iterations"] and s1["rel_change"] == s0["rel_change"]
    ctx.close()


@pytest.mark.parametrize("N,K,method,precision", [(64, 300, "fpsa", "mixed"), (64, 2000, "fpsa", "mixed"),
                                                  (64, 2000, "gmres", "mixed"), (56, 900, "fpsa", "mixed"),
                                                  (60, 900, "fpsa", "mixed"), (40, 700, "fpsa", "fp64"),
                                                  (44, 700, "fpsa", "fp64"), (40, 700, "gmres", "fp64"),
                                                  (32, 500, "fpsa", "mixed")])
def test_coarse_step(binding, N, K, method, precision):
    p = inputs.random_slab(K, N, N - 1, seed=1300 + K + N, kernel="srk", thick=(5, 200), c=(0.9, 0.999))
    kw = dict(inner_iterations=4) if precision == "mixed" and method == "fpsa" else {}
    _repeat(binding, p, 6, method, precision, **kw)


@pytest.mark.parametrize("N,K,R,precision", [(16, 64, 1, "fp64"), (16, 400, 2, "mixed"), (128, 40, 1, "mixed"),
                                             (64, 40, 3, "fp64")])
def test_solve_numbers(binding, N, K, R, precision):
    p = inputs.random_slab(K, N, N - 1, seed=1400 + K + N, kernel="hg", thick=(2, 60), c=(0.7, 0.99), nrhs=R)
    _repeat(binding, p, 30, "fpsa", precision, **(dict(inner_iterations=4) if precision == "mixed" else {}))


def test_engine_change(binding):
    import torch
    p = inputs.random_slab(90, 64, 63, seed=1500, kernel="hg", thick=(2, 60), c=(0.7, 0.99), nrhs=16)
    kw = dict(tol=1e-12, max_iterations=300, inner_iterations=4)
    ref = binding.context_for(p, laplacian="wfd", precision="mixed")
    ref.set_tuning({"solve_engine": 1})
    want, _ = ref.solve("fpsa", **kw)
    ref.close()
    busy = torch.ones((8192, 8192), device="cuda")
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        ctx = binding.context_for(p, laplacian="wfd", precision="mixed")
        ctx.solve("fpsa", **kw)
    torch.cuda.synchronize()
    for _ in range(20):
        busy = busy @ busy * 1e-4
    ctx.set_tuning({"solve_engine": 1})
    got, _ = ctx.solve("fpsa", **kw)
    ctx.close()
    assert np.array_equal(got, want)


@pytest.mark.parametrize("N,K,R", [(128, 200, 16), (128, 90, 64), (192, 60, 33), (256, 90, 16), (256, 40, 64)])
def test_tensor_core_pushes(binding, N, K, R):
    p = inputs.random_slab(K, N, N - 1, seed=1600 + K + N, kernel="hg", thick=(2, 60), c=(0.7, 0.99), nrhs=R)
    _repeat(binding, p, 6, "fpsa", "mixed", inner_iterations=4)
