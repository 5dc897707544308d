"""Contexts on a nearly full device. The BCR solve's own storage (the tensor-core solve's
copies of the factors, the dataflow solve's packets) is optional: a context that has no room
for it is created all the same and solves by the next form in the list, tensor cores,
dataflow, level by level. The last sums in the order of the dataflow solve's unstaged form
(2N above 128 in FP32), so against that one it gives the same bits (there is no coarse step
here). Otherwise the forms differ by rounding, which the iteration to 1e-12 removes
(c <= 0.99: errors below 1e-10, fluxes within 1e-9). The rest of the device is held by one
block while a context is made; all kernels involved have run before.
"""
import numpy as np
import pytest

from paper_1907_13013_gb300 import inputs

pytestmark = pytest.mark.gpu

MB = 1 << 20
KW = dict(tol=1e-12, max_iterations=300)


@pytest.fixture(scope="module")
def binding():
    import __graft_entry__ as g
    g.build()
    from paper_1907_13013_gb300 import binding as b
    return b


@pytest.fixture(autouse=True)
def give_back():
    """The held blocks go back to the device, not only to the caching allocator."""
    yield
    import torch
    torch.cuda.empty_cache()


def _free():
    import torch
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def _hold(leave):
    import torch
    return torch.empty(max(0, _free() - leave), dtype=torch.uint8, device="cuda")


def _usage(make):
    before = _free()
    ctx = make()
    used = before - _free()
    return ctx, used


def _bcr_launches(ctx, method, **kw):
    """Flux, statistics and the number of BCR solve kernels launched."""
    ctx.profile_enable(False)  # (resets the counters)
    phi, st = ctx.solve(method, **kw)
    return phi, st, ctx.profile_read()["bcr_solve"]["launches"]


@pytest.mark.parametrize("N,K,R,precision", [(16, 24000, 8, "fp64"), (128, 500, 16, "mixed"), (48, 900, 48, "mixed")])
def test_less_room_than_wanted(binding, N, K, R, precision):
    p = inputs.random_slab(K, N, N - 1, seed=1700 + N, kernel="hg", thick=(2, 60), c=(0.7, 0.99), nrhs=R)
    kw = dict(KW, inner_iterations=4) if precision == "mixed" else KW

    def make(engine=0):
        c = binding.context_for(p, laplacian="wfd", precision=precision)
        if engine:
            c.set_tuning({"solve_engine": engine})
        return c
    ctx, used = _usage(make)
    tensor = ctx.get_tuning()["solve_engine"] == 2
    want_tc = ctx.solve("fpsa", **kw)[0] if tensor else None
    ctx.set_tuning({"solve_engine": 1})
    want, _, plain = _bcr_launches(ctx, "fpsa", **kw)
    ctx.close()
    seen = set()
    leave, refused = used + 256 * MB, False
    while not refused and leave > 0:
        block = _hold(leave)
        try:
            ctx = make()
        except binding.FpsaError as err:
            assert "memory" in str(err)
            refused = True  # what a context cannot do without no longer fits
            del block
            continue
        engine = ctx.get_tuning()["solve_engine"]
        phi, _, launches = _bcr_launches(ctx, "fpsa", **kw)
        ctx.close()
        del block
        if engine == 2:
            seen.add("tensor")
            assert np.array_equal(phi, want_tc)
        elif launches <= plain:
            seen.add("dataflow")
            assert np.array_equal(phi, want)
        else:
            seen.add("levels")
            assert np.array_equal(phi, want) or N < 128
            assert np.abs(phi - want).max() / np.abs(want[..., 0]).max() < 1e-9
        leave -= max(8 * MB, used // 64)
    assert refused and "levels" in seen and (not tensor or "tensor" in seen)


def test_gmres_basis_takes_the_room(binding):
    N, K, R = 64, 2000, 16
    p = inputs.random_slab(K, N, N - 1, seed=1800, kernel="hg", thick=(2, 60), c=(0.7, 0.99), nrhs=R)
    kw = dict(tol=1e-10, max_iterations=100)
    ref, used = _usage(lambda: binding.context_for(p, laplacian="mpd", precision="mixed"))
    want, _ = ref.solve("gmres", **kw)
    basis = 34 * 4 * R * K * 2 * N
    ref.set_tuning({"solve_engine": 1})
    ref.solve("gmres", **kw)  # the dataflow kernels have run
    ref.close()
    block = _hold(used + basis - 64 * MB)
    ctx = binding.context_for(p, laplacian="mpd", precision="mixed")
    assert ctx.get_tuning()["solve_engine"] == 2
    got, _ = ctx.solve("gmres", **kw)
    assert ctx.get_tuning()["solve_engine"] == 1
    again, _ = ctx.solve("fpsa", tol=1e-12, max_iterations=300)  # and goes on working
    ctx.close()
    del block
    for x in (got, again):
        assert np.abs(x - want).max() / np.abs(want[..., 0]).max() < 1e-8
