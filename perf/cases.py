"""The solves and sweeps that the performance of this library is measured on.

Every case goes through the public entry points of paper_1907_13013_gb300: the
allocation-free sweep (binding.sweep_noalloc), a context's set_xs + solve on device
arrays, the differentiable solve (binding.FPSASolve) and the batch driver
(batch.BatchSolver, host arrays). One pass of a solve is what a program does for a new
set of cross sections: load and factorize them, then iterate to convergence.

The physics follows the workloads of inputs.py (Henyey-Greenstein and screened-
Rutherford slabs); each seed perturbs the cross sections of every cell, the sources and,
where the case says so, the cell widths, so that no two seeds are the same problem.
"""
import math
import random

import numpy as np
import torch

from paper_1907_13013_gb300 import batch, binding, inputs

_NOISE = 0.05  # relative spread of the seeded cross sections of the cells


def _solve(name, **kw):
    case = dict(name=name, kind="solve", precision="mixed", laplacian="wfd", method="fpsa", N=16, L=15, R=1, B=1,
                K=200, K_min=200, kernel="hg", shape=0.9, sigma_s0=100.0, sigma_a=1.0, source="uniform", beam=False,
                reflect=False, graded=False, tol=1e-10)
    case.update(kw)
    return case


def listed():
    return [
        # the smallest call: one sweep of a small slab, inside a caller's own iteration
        dict(name="sweep_small", kind="sweep", N=16, K=200),
        # the same entry point near its largest size
        dict(name="sweep_large", kind="sweep", N=64, K=2000),
        # plain source iteration in FP64 (the unaccelerated baseline of every comparison)
        _solve("plain_si", precision="fp64", method="si"),
        # the plain method: FPSA in FP64 on a small slab, MPD Laplacian
        _solve("plain_fpsa", precision="fp64", laplacian="mpd"),
        # FPSA-preconditioned GMRES in FP64 with a unit beam on a screened-Rutherford slab, L < N - 1
        _solve("beam_gmres", precision="fp64", laplacian="mpd", method="gmres", N=32, L=15, K=100, K_min=100,
               kernel="srk", shape=2.83e-5, beam=True, source="none"),
        # a few slabs of uneven size at once, several sources, graded cells, a symmetry plane on the left
        _solve("ragged_mixed", laplacian="mpd", N=32, L=31, R=3, B=6, K=613, K_min=37, shape=0.95, graded=True,
               reflect=True, source="random"),
        # one thick, strongly forward-peaked slab in mixed precision (the workload of bench.py)
        _solve("precision_mixed", N=64, L=63, K=2000, K_min=2000, kernel="srk", shape=1e-5, sigma_s0=1000.0,
               sigma_a=0.01, source="left_half"),
        # the same slab with everything in FP64
        _solve("precision_fp64", precision="fp64", N=64, L=63, K=2000, K_min=2000, kernel="srk", shape=1e-5,
               sigma_s0=1000.0, sigma_a=0.01, source="left_half"),
        # forward solve and gradients of a functional with respect to every cross section
        _solve("gradient", kind="gradient", laplacian="mpd", N=128, L=127, K=1000, K_min=1000, kernel="srk",
               shape=1e-6, sigma_s0=1000.0, sigma_a=0.01, tol=1e-12),
        # many right-hand sides of one large-order slab, the size of a shard of the scale workload
        _solve("scale_fpsa", laplacian="mpd", N=256, L=255, R=64, K=1250, K_min=1250, shape=0.99, sigma_s0=99.99,
               sigma_a=0.01, source="random"),
        # the same by GMRES-IR, fewer right-hand sides
        _solve("scale_gmres", laplacian="mpd", method="gmres", N=256, L=255, R=16, K=1250, K_min=1250, shape=0.99,
               sigma_s0=99.99, sigma_a=0.01, source="random"),
        # independent slabs of mixed orders and uneven sizes from host arrays, as one batch
        dict(name="batch", kind="batch", B=32, K_min=100, K=5000, sizes=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.choice(["sweep", "plain", "plain", "gmres", "mixed", "mixed", "mixed", "gradient", "many", "batch"])
    if what == "sweep":
        N = rng.choice([16, 32, 64, 128])
        return dict(kind="sweep", N=N, K=_log_int(rng, 50, 131072 // N))
    if what == "batch":
        return dict(kind="batch", B=rng.randint(8, 32), K_min=100, K=rng.randint(500, 4000), sizes=rng.randint(0, 9999))
    srk = rng.random() < 0.5
    kw = dict(kernel="srk" if srk else "hg",
              shape=math.exp(rng.uniform(math.log(1e-5), math.log(1e-4))) if srk else rng.uniform(0.8, 0.95),
              sigma_s0=math.exp(rng.uniform(math.log(50.0), math.log(1000.0))),
              sigma_a=math.exp(rng.uniform(math.log(0.01), math.log(1.0))), laplacian=rng.choice(["mpd", "wfd"]),
              source=rng.choice(["uniform", "left_half", "random"]), graded=rng.random() < 0.5)
    if what == "plain":
        N = rng.choice([16, 32, 64])
        kw.update(precision="fp64", N=N, K=_log_int(rng, 100, 64000 // N))
        if rng.random() < 0.3:
            kw.update(method="si", kernel="hg", shape=rng.uniform(0.8, 0.95), sigma_s0=rng.uniform(20.0, 100.0),
                      sigma_a=1.0)
        elif N < 64 and rng.random() < 0.4:
            kw.update(B=rng.randint(2, 8), R=rng.choice([1, 2]), K=kw["K"] // 4, reflect=rng.random() < 0.5)
    elif what == "gmres":
        N = rng.choice([16, 32, 64])
        kw.update(method="gmres", precision=rng.choice(["fp64", "mixed"]), N=N, K=_log_int(rng, 80, 32000 // N),
                  beam=rng.random() < 0.5, sigma_a=max(kw["sigma_a"], 0.1))
    elif what == "mixed":
        N = rng.choice([16, 32, 64, 128])
        kw.update(N=N, K=_log_int(rng, 100, 256000 // N))
        if rng.random() < 0.4:
            kw.update(B=rng.randint(2, 12), R=rng.randint(1, 5), K=max(40, kw["K"] // 5), reflect=rng.random() < 0.5,
                      beam=rng.random() < 0.3)
    elif what == "gradient":
        N = rng.choice([32, 64, 128])
        kw.update(kind="gradient", N=N, K=_log_int(rng, 100, 128000 // N), tol=1e-12)
    else:
        N = rng.choice([64, 128, 256])
        kw.update(N=N, R=rng.randint(16, 64), K=_log_int(rng, 200, 240000 // N), kernel="hg",
                  shape=rng.uniform(0.8, 0.99), source="random", laplacian="mpd")
    kw["L"] = kw["N"] - 1
    kw["K_min"] = max(1, kw["K"] // 9) if kw.get("B", 1) > 1 else kw["K"]
    case = _solve("", **kw)
    del case["name"]
    return case


def _cells(case):
    """Cell counts of the instances: from the largest down to the smallest."""
    B, K, lo = case["B"], case["K"], case["K_min"]
    return [K] if B == 1 else [K - (K - lo) * b // (B - 1) for b in range(B)]


def _batch_sizes(case):
    r = random.Random(case["sizes"])
    return [(r.randint(case["K_min"], case["K"]), r.choice([16, 32, 64, 128])) for _ in range(case["B"])]


def _quadrature(N):
    mu, w = np.polynomial.legendre.leggauss(N)
    return mu, w


def _fields(case, seed):
    """Host arrays of one context's problem: h, sigma_t, sigma_s, source [R][sumK][2] (moment 0), incident."""
    rng = np.random.default_rng(seed)
    Ks, L, R = _cells(case), case["L"], case["R"]
    n = sum(Ks)
    f = inputs.srk_moments(case["shape"], L) if case["kernel"] == "srk" else inputs.hg_moments(case["shape"], L)
    s0 = case["sigma_s0"] * np.exp(_NOISE * rng.standard_normal(n))
    sa = case["sigma_a"] * np.exp(_NOISE * rng.standard_normal(n))
    widths = []
    for K in Ks:
        x = rng.uniform(0.5, 1.5, K) if case["graded"] else np.ones(K)
        widths.append(x / x.sum())
    src = rng.uniform(0.5, 1.0, (R, 1, 1)) * np.ones((R, n, 2))
    if case["source"] == "random":
        src = rng.uniform(0.0, 1.0, (R, n, 2))
    elif case["source"] == "left_half":
        at = np.concatenate([np.arange(K) < max(1, K // 2) for K in Ks])
        src = src * at[None, :, None]
    elif case["source"] == "none":
        src = src * 0.0
    inc = None
    if case["beam"]:
        mu, w = _quadrature(case["N"])
        inc = np.zeros((R, len(Ks), 2, case["N"]))
        inc[:, :, 0, -1] = rng.uniform(0.5, 1.0, (R, len(Ks))) / (w[-1] * mu[-1])
    return dict(h=np.concatenate(widths), sigma_t=sa + s0, sigma_s=s0[:, None] * f[None], src=src, inc=inc)


def _dev(x):
    return torch.as_tensor(x, dtype=torch.float64).cuda()


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    if case["kind"] == "sweep":
        K, N = case["K"], case["N"]
        x = rng.uniform(0.5, 1.5, K)
        return dict(case=case, h=_dev(x / x.sum()), sigma_t=_dev(np.exp(rng.uniform(np.log(10.0), np.log(300.0), K))),
                    q=_dev(rng.uniform(0.0, 1.0, (K, 2, N))), psi=torch.zeros((K, 2, N), dtype=torch.float64).cuda())
    if case["kind"] == "batch":
        return dict(case=case, problems=_batch_problems(case, seed))
    f = _fields(case, seed)
    bc = ("reflective", "vacuum") if case["reflect"] else None
    ctx = binding.Context(_cells(case), f["h"], case["N"], case["L"], n_rhs=case["R"], laplacian=case["laplacian"],
                          precision=case["precision"], bc=bc)
    if f["inc"] is not None:
        ctx.set_incident(_dev(f["inc"]))
    q = torch.zeros(f["src"].shape + (case["L"] + 1,), dtype=torch.float64, device="cuda")
    q[..., 0] = _dev(f["src"])
    state = dict(case=case, ctx=ctx, sigma_t=_dev(f["sigma_t"]), sigma_s=_dev(f["sigma_s"]), q=q)
    if case["kind"] == "gradient":
        state["sigma_t"].requires_grad_()
        state["sigma_s"].requires_grad_()
        state["weight"] = _dev(_weight(case, seed))
    else:
        state["phi"] = torch.zeros_like(q)
    return state


def _weight(case, seed):
    """d(objective)/d(phi): a detector response on the scalar flux and the current."""
    rng = np.random.default_rng(seed + 1)
    g = np.zeros((case["R"], sum(_cells(case)), 2, case["L"] + 1))
    g[..., 0] = rng.uniform(0.0, 1.0, g.shape[:-1])
    g[..., 1] = rng.uniform(-0.5, 0.5, g.shape[:-1])
    return g


def _batch_problems(case, seed):
    rng = np.random.default_rng(seed)
    out = []
    for K, N in _batch_sizes(case):
        g, c = rng.uniform(0.8, 0.99, 2), rng.uniform(0.9, 0.999, 2)
        st = np.exp(rng.uniform(0.0, np.log(1000.0), 2))
        reg = (np.arange(K) >= K // 2).astype(int)
        ss = (c * st)[reg][:, None] * np.stack([inputs.hg_moments(x, N - 1) for x in g])[reg]
        out.append(inputs.slab(K, N, N - 1, 1.0, st[reg], ss, 1.0))
    return out


def run(state):
    case = state["case"]
    if case["kind"] == "sweep":
        return binding.sweep_noalloc(case["N"], state["h"], state["sigma_t"], state["q"], state["psi"])
    if case["kind"] == "batch":
        return batch.BatchSolver(state["problems"], graph=True).solve(tol=1e-10, max_iterations=200)[0]
    if case["kind"] == "gradient":
        phi = binding.FPSASolve.apply(state["ctx"], state["sigma_t"], state["sigma_s"], state["q"], case["tol"])
        d_st, d_ss = torch.autograd.grad(phi, (state["sigma_t"], state["sigma_s"]), state["weight"])
        return phi.detach(), d_st, d_ss
    state["ctx"].set_xs(state["sigma_t"], state["sigma_s"], state["q"])
    return state["ctx"].solve(case["method"], tol=case["tol"], out=state["phi"])[0]


def _method_work(cells, N, L1, R, method, passes):
    """Bytes in and out of a solve; operations of its factorization and of `passes` iterations."""
    sweeps = {"si": 1000, "fpsa": 20, "gmres": 12}[method] * passes
    nbytes = 8.0 * cells * (2 + L1 + 4 * R * L1)
    contractions = 16.0 * N * L1 if method != "si" else 8.0 * N * L1
    correction = 12.0 * N * N if method != "si" else 0.0
    factor = 2.0 * (2 * N) ** 3 if method != "si" else 0.0
    return nbytes, cells * (factor + R * sweeps * (contractions + correction + 28.0 * N))


def work(case):
    if case["kind"] == "sweep":
        return {"bytes": 8.0 * case["K"] * (2 + 4 * case["N"]), "flops": 28.0 * case["K"] * case["N"]}
    if case["kind"] == "batch":
        parts = [_method_work(K, N, N, 1, "fpsa", 1) for K, N in _batch_sizes(case)]
    else:
        passes = 2 if case["kind"] == "gradient" else 1
        parts = [_method_work(sum(_cells(case)), case["N"], case["L"] + 1, case["R"], case["method"], passes)]
    nbytes, flops = (sum(p[k] for p in parts) for k in (0, 1))
    if case["kind"] == "gradient":
        nbytes += 8.0 * sum(_cells(case)) * (2 + 3 * (case["L"] + 1))
    return {"bytes": nbytes, "flops": flops}


# ---- the discrete solutions in 64 bits, by a direct method (numpy and torch only)


def _operators(N, L):
    mu, w = _quadrature(N)
    P = np.polynomial.legendre.legvander(mu, L)                      # [n][l]
    return mu, (w[:, None] * P).T, (np.arange(L + 1) + 0.5) * P      # mu, D [l][n], M [n][l]


def _streaming(mu):
    """[a][b][n]: the upwind streaming part of a cell's 2 x 2 node block."""
    neg, pos = mu < 0, mu > 0
    return np.array([[0.5 * mu - mu * neg, 0.5 * mu], [-0.5 * mu, -0.5 * mu + mu * pos]])


def _blocks(mu, D, M, h, st, ss, reflect):
    """Diagonal blocks of the discrete transport operator [K][2N][2N] and its coupling blocks to the left and right."""
    N, K = mu.size, h.numel()
    dev = h.device
    t = lambda x: torch.as_tensor(x, dtype=torch.float64, device=dev)  # noqa: E731
    S = torch.einsum("nl,kl,lm->knm", t(M), ss, t(D))
    own = st[:, None, None] * torch.eye(N, dtype=torch.float64, device=dev) - S
    G = t(_streaming(mu))
    A = torch.empty((K, 2, N, 2, N), dtype=torch.float64, device=dev)
    for a in range(2):
        for b in range(2):
            A[:, a, :, b, :] = (h / (3.0 if a == b else 6.0))[:, None, None] * own + torch.diag(G[a, b])
    m = t(mu)
    i = torch.arange(N, device=dev)
    if reflect:  # the left edge mirrors: incoming mu > 0 is the outgoing -mu
        p = i[m > 0]
        A[0, 0, p, 0, N - 1 - p] -= m[p]
    left, right = torch.zeros((2, N, 2, N), dtype=torch.float64, device=dev), torch.zeros(
        (2, N, 2, N), dtype=torch.float64, device=dev)
    left[0, i, 1, i] = -m.clamp(min=0.0)
    right[1, i, 0, i] = m.clamp(max=0.0)
    n2 = 2 * N
    A = A.reshape(K, n2, n2)
    Lc = left.reshape(1, n2, n2).repeat(K, 1, 1)
    Rc = right.reshape(1, n2, n2).repeat(K, 1, 1)
    Lc[0] = 0.0
    Rc[-1] = 0.0
    return A, Lc, Rc


def _block_solve(A, Lc, Rc, r):
    """Block tridiagonal solve, A [K][n][n], couplings to k - 1 and k + 1, r [K][n][m]: odd cells eliminated first."""
    K, n = A.shape[0], A.shape[1]
    if K == 1:
        return torch.linalg.solve(A, r)
    X = torch.linalg.solve(A[1::2], torch.cat([Lc[1::2], Rc[1::2], r[1::2]], dim=2))
    XL, XR, xr = X[:, :, :n], X[:, :, n:2 * n], X[:, :, 2 * n:]
    Ae, re, ne = A[0::2].clone(), r[0::2].clone(), (K + 1) // 2
    Le, Re = torch.zeros_like(Ae), torch.zeros_like(Ae)
    no = K // 2                        # the odd cell 2 j + 1 lies between the even ones j and j + 1
    lo = Lc[2::2]                      # couplings of the even cells 1 .. to their left odd neighbour
    Ae[1:] -= lo @ XR[:ne - 1]
    re[1:] -= lo @ xr[:ne - 1]
    Le[1:] = -(lo @ XL[:ne - 1])
    ro = Rc[0::2][:no]                 # couplings of the even cells to their right odd neighbour
    Ae[:no] -= ro @ XL
    re[:no] -= ro @ xr
    Re[:no] = -(ro @ XR)
    ue = _block_solve(Ae, Le, Re, re)
    uo = xr - XL @ ue[:no]
    uo[:ne - 1] -= XR[:ne - 1] @ ue[1:]
    u = torch.empty_like(r)
    u[0::2] = ue
    u[1::2] = uo
    return u


def _direct(N, L, h, st, ss, src, inc=None, reflect=False, weight=None):
    """phi [R][K][2][L+1] of one slab (src: moment 0 of the source, [R][K][2]) and, with `weight` = d(objective)/d(phi),
    the gradients with respect to sigma_t and sigma_s."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    t = lambda x: torch.as_tensor(x, dtype=torch.float64, device=dev)  # noqa: E731
    mu, D, M = _operators(N, L)
    h, st, ss, src = t(h), t(st), t(ss), t(src)
    K, R = h.numel(), src.shape[0]
    A, Lc, Rc = _blocks(mu, D, M, h, st, ss, reflect)
    q = src[..., None] * t(M[:, 0])                                   # [R][K][2][N]
    r = _mass(h, q)
    if inc is not None:
        m, g = t(mu), t(inc)                                          # [R][2][N]
        if not reflect:
            r[:, 0, 0] += m.clamp(min=0.0) * g[:, 0]
        r[:, -1, 1] -= m.clamp(max=0.0) * g[:, 1]
    psi = _block_solve(A, Lc, Rc, r.reshape(R, K, 2 * N).permute(1, 2, 0)).permute(2, 0, 1).reshape(R, K, 2, N)
    phi = psi @ t(D).T
    if weight is None:
        return phi
    # A^T lambda = D^T weight; d/d(sigma_t) = -lambda m psi, d/d(sigma_s,l) = lambda m M_l phi_l
    At = A.transpose(1, 2)
    Lt, Rt = torch.zeros_like(Lc), torch.zeros_like(Rc)
    Lt[1:] = Rc[:-1].transpose(1, 2)
    Rt[:-1] = Lc[1:].transpose(1, 2)
    s = (t(weight) @ t(D)).reshape(R, K, 2 * N).permute(1, 2, 0)
    lam = _block_solve(At, Lt, Rt, s).permute(2, 0, 1).reshape(R, K, 2, N)
    d_st = -(lam * _mass(h, psi)).sum(dim=(0, 2, 3))
    d_ss = ((lam @ t(M)) * _mass(h, phi)).sum(dim=(0, 2))
    return phi, d_st, d_ss


def _mass(h, x):
    """The cells' mass matrix on the node axis of x [R][K][2][...]."""
    w = (h / 6.0)[None, :, None]
    return torch.stack([w * (2.0 * x[:, :, 0] + x[:, :, 1]), w * (x[:, :, 0] + 2.0 * x[:, :, 1])], dim=2)


def _exact_sweep(case, seed):
    s = prepare(case, seed)
    mu, _ = _quadrature(case["N"])
    h, st, q = (s[k].cpu().numpy() for k in ("h", "sigma_t", "q"))
    G, psi = _streaming(mu), np.zeros_like(q)
    pos, flow = mu > 0, np.zeros(mu.size)
    K = h.size
    for p in range(K):
        c = np.where(pos, p, K - 1 - p)       # each direction in its own order of cells
        hh, sg, i = h[c], st[c], np.arange(mu.size)
        q0, q1 = q[c, 0, i], q[c, 1, i]
        r0 = hh / 6.0 * (2.0 * q0 + q1) + np.where(pos, mu * flow, 0.0)
        r1 = hh / 6.0 * (q0 + 2.0 * q1) - np.where(pos, 0.0, mu * flow)
        T = [[G[a, b] + sg * hh / (3.0 if a == b else 6.0) for b in range(2)] for a in range(2)]
        det = T[0][0] * T[1][1] - T[0][1] * T[1][0]
        x0, x1 = (r0 * T[1][1] - T[0][1] * r1) / det, (T[0][0] * r1 - T[1][0] * r0) / det
        psi[c, 0, i], psi[c, 1, i] = x0, x1
        flow = np.where(pos, x1, x0)
    return psi


def exact(case, seed):
    if case["kind"] == "sweep":
        return _exact_sweep(case, seed)
    if case["kind"] == "batch":
        out, spent = [], 0.0
        for p in _batch_problems(case, seed):
            cost = p["h"].size * (2.0 * p["N"]) ** 3
            if spent + cost > 2e11:  # the direct solution of all the large ones would take too long
                out.append(None)
                continue
            spent += cost
            out.append(_direct(p["N"], p["L"], p["h"], p["sigma_t"], p["sigma_s"], p["Q"][None, :, :, 0])[0]
                       .cpu().numpy())
        return out
    f = _fields(case, seed)
    if case["kind"] == "gradient":
        if case["B"] != 1:
            return None
        return _direct(case["N"], case["L"], f["h"], f["sigma_t"], f["sigma_s"], f["src"], weight=_weight(case, seed))
    parts, o = [], 0
    for b, K in enumerate(_cells(case)):
        at = slice(o, o + K)
        o += K
        parts.append(_direct(case["N"], case["L"], f["h"][at], f["sigma_t"][at], f["sigma_s"][at], f["src"][:, at],
                             inc=None if f["inc"] is None else f["inc"][:, b], reflect=case["reflect"]))
    return torch.cat(parts, dim=1)
