"""The convergence test with untested iterations between the tests (check_every): a test sees
the largest change and the largest flux since the one before it, the last iteration allowed
is tested in any case, and the flux returned is the iterate after exactly the iterations
reported (an iteration launched behind the last report leaves it alone). Compared with the
oracle's iterates after that many iterations; both sides compute in FP64, a fixed number of
contracting iterations of at most some hundred operations a value: 1e-9 of the largest flux
is far above their rounding, and far below the change of one iteration here.
"""
import numpy as np
import pytest

from oracle import iterations as oit
from paper_1907_13013_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method", ["si", "fpsa"])
@pytest.mark.parametrize("every,tol,limit", [(3, 1e-5, 1000), (3, 0.0, 7), (4, 0.0, 8), (5, 1e-3, 1000), (1, 1e-4, 1000)])
def test_untested_iterations(method, every, tol, limit):
    import torch  # noqa: F401
    import __graft_entry__ as g
    g.build()
    from paper_1907_13013_gb300 import binding
    p = inputs.random_slab(23, 16, 15, seed=2000, kernel="hg", thick=(2, 20), c=(0.6, 0.9))

    def iterate(n):
        if n == 0:
            return np.zeros((23, 2, 16))
        if method == "si":
            return oit.source_iteration(p, tol=0.0, max_it=n)[0]
        return oit.fpsa_source_iteration(p, "mpd", tol=0.0, max_it=n)[0]
    n, change, flux, last = 0, 0.0, 0.0, iterate(0)
    while True:
        n += 1
        phi = iterate(n)
        change = max(change, np.abs(phi[..., 0] - last[..., 0]).max())
        flux = max(flux, np.abs(phi[..., 0]).max())
        last = phi
        if n % every and n < limit:
            continue
        e = change / flux
        if e < tol or n == limit:
            break
        change = flux = 0.0
    ctx = binding.context_for(p, laplacian="mpd", precision="fp64")
    got, st = ctx.solve(method, tol=tol, max_iterations=limit, check_every=every, raise_on_notconv=False)
    ctx.close()
    assert st["iterations"] == n and st["sweeps"] == n
    assert (st["status"] == 0) == (e < tol)
    assert abs(st["rel_change"] - e) < 1e-9
    assert np.abs(got[0] - last).max() / np.abs(last[..., 0]).max() < 1e-9
