"""Workloads of the implicit DG solver that its speed is judged on.

A case is one call (or one short sequence of calls) through the package's public entry points: assembly, block SpMV,
factorization, preconditioner apply, preconditioned solve, differentiable solve, batched solve and pseudo-time march.
Inputs are seeded synthetic O-grids around a NACA-like curve with a perturbed free stream, drawn here on the GPU; sizes
follow the repository's workload configurations (16 x 8 p=1 up to 256 x 128 p=3) and odd sizes between them.

Solves run to a relative residual of 1e-10 (the default of the differentiable solve and of the march) or tighter, so
that a solution is fixed well beyond the digits in which two correct factorizations of one matrix differ.
"""
import math

import numpy as np
import torch

import paper_2101_01763_gb300 as sg

GAMMA = 1.4
DEV = "cuda"


# ------------------------------------------------------------------------------------------------ the cases
def _grid(kind, p, n_theta, n_r, **more):
    return dict(kind=kind, p=p, n_theta=n_theta, n_r=n_r, **more)


def listed():
    return [
        # one Newton step's linear solve on the smallest grid: launches and host round trips count
        dict(name="factor_solve_16x8_p1", **_grid("factor_solve", 1, 16, 8, precision="mixed", eps=1e-2, s=4,
                                                  restart=40, tol=1e-10, mach=0.5, amp=0.05, cfl=10.0)),
        # the ordinary Newton step: p=2 on a 64 x 32 grid, factors in FP32 refined by the FP64 outer solve
        dict(name="factor_solve_64x32_p2", **_grid("factor_solve", 2, 64, 32, precision="mixed", eps=1e-3, s=4,
                                                   restart=60, tol=1e-10, mach=0.5, amp=0.05, cfl=10.0)),
        # the same step with every factor in FP64 (the default precision of the factorization)
        dict(name="factor_solve_64x32_p2_fp64", **_grid("factor_solve", 2, 64, 32, precision="fp64", eps=1e-3, s=4,
                                                        restart=60, tol=1e-10, mach=0.5, amp=0.05, cfl=10.0)),
        # the largest Newton step of one GPU: p=3 on 256 x 128, 2.1 million unknowns
        dict(name="factor_solve_256x128_p3", **_grid("factor_solve", 3, 256, 128, precision="mixed", eps=1e-3, s=8,
                                                     restart=80, tol=1e-10, mach=0.8, amp=0.1, cfl=10.0)),
        # many independent flow conditions solved together (grids 32 x 16 to 96 x 48, p = 1..3)
        dict(name="batched_8", kind="batched", systems=8, largest=96, precision="mixed", eps=1e-3, s=4, restart=60,
             tol=1e-10),
        # a gradient step through the solve: forward, transposed solve, dL/dA on the block pattern; an odd grid
        dict(name="adjoint_80x41_p2", **_grid("adjoint", 2, 80, 41, precision="mixed", eps=1e-3, s=4, restart=60,
                                              tol=1e-10, mach=0.5, amp=0.05, cfl=10.0)),
        # repeated right-hand sides with a factor in hand, loose tolerance (eps = 0.1): applies and SpMVs dominate
        dict(name="solve_192x96_p3", **_grid("solve", 3, 192, 96, precision="mixed", eps=1e-1, s=4, restart=60,
                                             tol=1e-10, mach=0.6, amp=0.05, cfl=10.0, transpose=False)),
        # a weak preconditioner at a large time step: many columns, Gram reductions and block updates; transposed
        dict(name="solve_weak_75x33_p3", **_grid("solve", 3, 75, 33, precision="mixed", eps=0.5, s=8, restart=80,
                                                 tol=1e-12, mach=0.5, amp=0.05, cfl=100.0, transpose=True)),
        # the preconditioner alone in FP64, as an outer solver of the user's own calls it, both directions
        dict(name="apply_64x32_p2_fp64", **_grid("apply", 2, 64, 32, eps=1e-3, mach=0.5, amp=0.05, cfl=10.0)),
        # the matrix alone, both directions, at the largest size (5.35 GB of blocks)
        dict(name="spmv_256x128_p3", **_grid("spmv", 3, 256, 128, mach=0.8, amp=0.1, cfl=10.0)),
        # residual and exact Jacobian at the largest size
        dict(name="assemble_256x128_p3", **_grid("assemble", 3, 256, 128, mach=0.8, amp=0.1, cfl=10.0, bc="wall")),
        # pseudo-time continuation with the CFL ramp on a small odd grid
        dict(name="march_50x23_p1", **_grid("march", 1, 50, 23, precision="mixed", eps=1e-3, s=4, restart=60,
                                            tol=1e-10, mach=0.5, amp=0.05, cfl=10.0, steps=3)),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_grid(rng, kind, most, **more):
    """A grid of p, n_theta and n_r (any parity) of at most `most` unknowns."""
    while True:
        p, n_theta, n_r = rng.randint(1, 3), _log_int(rng, 12, 256), _log_int(rng, 6, 128)
        if n_theta * n_r * 4 * (p + 1) ** 2 <= most and n_r <= n_theta <= 6 * n_r:
            return _grid(kind, p, n_theta, n_r, mach=round(rng.uniform(0.3, 0.8), 3),
                         amp=rng.choice([0.05, 0.1]), cfl=10.0, **more)


def draw(rng):
    kind = rng.choice(["factor_solve"] * 4 + ["factor_solve_fp64", "solve", "solve_weak", "adjoint", "apply", "spmv",
                                              "assemble", "march", "batched"])
    s = rng.choice([4, 8])
    opts = dict(precision="mixed", s=s, restart=s * rng.randint(8, 15), tol=1e-10)
    if kind == "factor_solve":
        return _draw_grid(rng, kind, 1_300_000, eps=rng.choice([1e-2, 1e-3]), **opts)
    if kind == "factor_solve_fp64":
        return _draw_grid(rng, "factor_solve", 80_000, eps=rng.choice([1e-2, 1e-3]), **dict(opts, precision="fp64"))
    if kind == "solve":
        return _draw_grid(rng, kind, 1_300_000, eps=rng.choice([1e-1, 1e-2]), transpose=rng.random() < 0.5, **opts)
    if kind == "solve_weak":
        return dict(_draw_grid(rng, "solve", 160_000, eps=0.5, transpose=rng.random() < 0.5,
                               **dict(opts, tol=1e-12)), cfl=100.0)
    if kind == "adjoint":
        return _draw_grid(rng, kind, 130_000, eps=1e-3, **opts)
    if kind == "apply":
        return _draw_grid(rng, kind, 80_000, eps=rng.choice([0.0, 1e-3, 1e-2]))
    if kind == "spmv":
        return _draw_grid(rng, kind, 2_100_000)
    if kind == "assemble":
        return _draw_grid(rng, kind, 2_100_000, bc=rng.choice(["wall", "farfield"]))
    if kind == "march":
        return _draw_grid(rng, kind, 50_000, eps=1e-3, steps=rng.randint(2, 4), **opts)
    return dict(kind="batched", systems=rng.randint(2, 8), largest=rng.choice([32, 64, 96]), eps=1e-3, **opts)


def _systems(case):
    """The systems of a batched case: its grids, degrees and flows follow from the number of systems alone."""
    r = np.random.RandomState(2101 + case["systems"])
    grids = [g for g in ((32, 16), (64, 32), (96, 48)) if g[0] <= case["largest"]]
    out = []
    for q in range(case["systems"]):
        n_theta, n_r = grids[(q + 1) % len(grids)]
        out.append(dict(p=1 + (q + q // 3) % 3, n_theta=n_theta, n_r=n_r, mach=float(r.uniform(0.3, 0.8)), amp=0.05,
                        cfl=10.0))
    return out


# ------------------------------------------------------------------------------------------------ seeded inputs
def _mesh(n_theta, n_r, gen):
    """Nodes [n_r + 1, n_theta, 2] of an O-grid from a NACA-0012-like curve to a circle of 20 chords; inner nodes
    moved by up to a tenth of their shortest edge."""
    phi = 2 * math.pi * torch.arange(n_theta, dtype=torch.float64) / n_theta
    x = 0.5 * (1 + torch.cos(phi))
    half = 0.6 * (0.2969 * x.clamp(min=0).sqrt() - 0.1260 * x - 0.3516 * x**2 + 0.2843 * x**3 - 0.1036 * x**4)
    sn = torch.sin(phi)
    sn[sn.abs() < 1e-14] = 0.0
    inner = torch.stack([x, -torch.sign(sn) * half], -1)
    outer = torch.stack([0.5 + 20 * torch.cos(phi), -20 * torch.sin(phi)], -1)
    g = 1 + 4.0 / n_r
    t = (g ** torch.arange(n_r + 1, dtype=torch.float64) - 1) / (g**n_r - 1)
    X = inner[None] + t[:, None, None] * (outer - inner)[None]
    C = X[1:n_r]
    edge = torch.stack([(X[2:] - C).norm(dim=-1), (X[:-2] - C).norm(dim=-1), (C.roll(-1, 1) - C).norm(dim=-1),
                        (C.roll(1, 1) - C).norm(dim=-1)]).amin(0)
    X[1:n_r] = C + (0.2 * torch.rand(C.shape, generator=gen, dtype=torch.float64) - 0.1) * edge[..., None]
    return X


def _state(X, c, gen):
    """Modal state [K, (p+1)^2, 4]: free stream with four smooth fields of relative size amp and small higher modes."""
    n_r, p, mach, amp = X.shape[0] - 1, c["p"], c["mach"], c["amp"]
    cen = 0.25 * (X[:n_r] + X[:n_r].roll(-1, 1) + X[1:] + X[1:].roll(-1, 1)).reshape(-1, 2)

    def smooth():
        k, th, ph, a = (torch.rand((4, 4), generator=gen, dtype=torch.float64))
        k, th, ph, a = 0.3 + 2.7 * k, 2 * math.pi * th, 2 * math.pi * ph, 0.5 + 0.5 * a
        arg = cen[:, :1] * (k * torch.cos(th)) + cen[:, 1:] * (k * torch.sin(th)) + ph
        return (a * torch.sin(arg)).sum(1) / a.sum()

    al = math.radians(2.0)
    rho = 1 + amp * smooth()
    u = mach * math.cos(al) * (1 + amp * smooth())
    v = mach * (math.sin(al) + amp * smooth())
    pr = (1 + amp * smooth()) / GAMMA
    uh = torch.zeros((cen.shape[0], (p + 1) ** 2, 4), dtype=torch.float64)
    uh[:, 0] = 2 * torch.stack([rho, rho * u, rho * v, pr / (GAMMA - 1) + 0.5 * rho * (u * u + v * v)], -1)
    size = 0.2 * amp * torch.tensor([1.0, mach, mach, 1 / (GAMMA - 1)], dtype=torch.float64)
    for m in range(1, (p + 1) ** 2):
        z = torch.randn((cen.shape[0], 4), generator=gen, dtype=torch.float64).clamp(-2, 2)
        uh[:, m] = size * z / (1 + m % (p + 1) + m // (p + 1))
    return uh


def _inputs(c, seed):
    gen = torch.Generator().manual_seed(seed)
    X = _mesh(c["n_theta"], c["n_r"], gen)
    return X.to(DEV), _state(X, c, gen).to(DEV)


def _vector(n, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed + 77)
    return torch.randn(n, generator=gen, dtype=torch.float64, device=DEV)


def _assemble(c, X, u):
    return sg.assemble(X, c["p"], u, c["mach"], 2.0, c["cfl"], bc=c.get("bc", "wall"))


def _block(c):
    return 4 * (c["p"] + 1) ** 2


# ------------------------------------------------------------------------------------------------ the calls
def prepare(case, seed):
    st = dict(case=case)
    kind = case["kind"]
    if kind == "batched":
        st["systems"] = _systems(case)
        for key in ("A", "b", "plan"):
            st[key] = []
        for q, c in enumerate(st["systems"]):
            rhs, A, _ = _assemble(c, *_inputs(c, 1000 * seed + q))
            st["A"].append(A)
            st["b"].append(rhs)
            st["plan"].append(sg.Plan(c["n_theta"], c["n_r"], _block(c)))
        return st
    X, u = _inputs(case, seed)
    if kind in ("assemble", "march"):
        st.update(X=X, u=u)
    if kind == "march":
        st["plan"] = sg.Plan(case["n_theta"], case["n_r"], _block(case))
    if kind in ("assemble", "march"):
        return st
    st["b"], st["A"], _ = _assemble(case, X, u)
    if kind in ("spmv", "apply", "adjoint"):
        st["x"] = _vector(st["b"].numel(), seed)
    if kind == "spmv":
        return st
    st["plan"] = sg.Plan(case["n_theta"], case["n_r"], _block(case))
    if kind == "solve":
        st["F"] = sg.Factor(st["plan"], st["A"], case["eps"], case["precision"])
    if kind == "apply":
        st["F"] = sg.Factor(st["plan"], st["A"], case["eps"], "fp64")
    return st


def run(state):
    c = state["case"]
    kind = c["kind"]
    if kind == "spmv":
        return [sg.spmv(state["A"], state["x"]), sg.spmv(state["A"], state["x"], transpose=True)]
    if kind == "assemble":
        rhs, A, dtau = _assemble(c, state["X"], state["u"])
        return [rhs, A.val, dtau]
    if kind == "apply":
        return [state["F"].apply(state["x"]), state["F"].apply(state["x"], transpose=True)]
    opts = dict(s=c["s"], restart=c["restart"], tol=c["tol"])
    if kind == "factor_solve":
        F = sg.Factor(state["plan"], state["A"], c["eps"], c["precision"])
        return sg.sstep_gmres(state["A"], F, state["b"], max_iters=600, **opts)[0]
    if kind == "solve":
        return sg.sstep_gmres(state["A"], state["F"], state["b"], max_iters=600, transpose=c["transpose"], **opts)[0]
    if kind == "adjoint":
        val, b = state["A"].val.detach().requires_grad_(), state["b"].detach().requires_grad_()
        x = sg.SpandSolve.apply(val, b, state["A"], state["plan"], c["eps"], c["precision"], c["s"], c["restart"],
                                c["tol"])
        return [x.detach(), *torch.autograd.grad(x, (val, b), state["x"])]
    if kind == "march":
        u, h = sg.march(state["X"], c["p"], state["u"], c["mach"], 2.0, state["plan"], cfl0=c["cfl"],
                        max_steps=c["steps"], eps=c["eps"], precision=c["precision"], **opts)
        return [u, h["res"], h["cfl"], h["dtau"]]
    Fs = sg.factor_batched(state["plan"], state["A"], c["eps"], c["precision"])
    return sg.sstep_gmres_batched(state["A"], Fs, state["b"], **opts)[0]


# ------------------------------------------------------------------------------------------------ what a pass needs
def _nnzb(c):
    return 5 * c["n_theta"] * c["n_r"] - 2 * c["n_theta"]


def _factor_flops(c):
    """Dense work of the leaf level alone: boxes of about 32 elements (their LU, the two triangular products with the
    24 elements around each and the Schur update).  The levels above add an amount that depends on the ranks."""
    n, m, boxes = 32 * _block(c), 24 * _block(c), c["n_theta"] * c["n_r"] / 32
    return boxes * (2 / 3 * n**3 + 2 * n * n * m + 2 * n * m * m)


def work(case):
    kind = case["kind"]
    if kind == "batched":
        ones = [work(dict(c, kind="factor_solve")) for c in _systems(case)]
        return {k: sum(w[k] for w in ones) for k in ("bytes", "flops")}
    B, nnzb = _block(case), _nnzb(case)
    N = case["n_theta"] * case["n_r"] * B
    mat, spmv = 8 * nnzb * B * B, 2 * nnzb * B * B
    if kind == "spmv":
        return {"bytes": 2 * mat + 32 * N, "flops": 2 * spmv}
    if kind == "assemble":
        q = case["p"] + 2
        # per quadrature point: the products of test functions, 4 x 4 flux Jacobian and trial functions
        points = q * q + 4 * q * 2
        return {"bytes": mat + 16 * N, "flops": case["n_theta"] * case["n_r"] * points * 2 * B * B}
    if kind == "apply":
        # the factor is read once for each direction; it is at least as large as the matrix
        return {"bytes": 2 * mat + 32 * N, "flops": 2 * spmv}
    if kind == "solve":
        # at least one column: the matrix and the factor (at least as large as the matrix in its own precision)
        return {"bytes": mat + mat / 2 + 16 * N, "flops": 2 * spmv}
    if kind == "adjoint":
        return {"bytes": 2 * mat + 32 * N, "flops": _factor_flops(case) + 4 * spmv}
    if kind == "march":
        return {"bytes": case["steps"] * 2 * mat + 16 * N, "flops": case["steps"] * _factor_flops(case)}
    return {"bytes": mat + 16 * N, "flops": _factor_flops(case) + 2 * spmv}


# ------------------------------------------------------------------------------------------------ in 64 bits
def _legendre(p, t):
    """Values and derivatives [len(t), p + 1] of the orthonormal Legendre polynomials."""
    V, D = np.zeros((len(t), p + 1)), np.zeros((len(t), p + 1))
    for a in range(p + 1):
        coef = np.zeros(a + 1)
        coef[a] = math.sqrt((2 * a + 1) / 2)
        V[:, a] = np.polynomial.legendre.legval(t, coef)
        if a:
            D[:, a] = np.polynomial.legendre.legval(t, np.polynomial.legendre.legder(coef))
    return torch.as_tensor(V, device=DEV), torch.as_tensor(D, device=DEV)


def _flux(U, n):
    rho, m, E = U[0], U[1:3], U[3]
    vn = (m @ n) / rho
    pr = (GAMMA - 1) * (E - 0.5 * (m @ m) / rho)
    return torch.cat([(rho * vn)[None], m * vn + pr * n, ((E + pr) * vn)[None]])


def _speed(U, n):
    pr = (GAMMA - 1) * (U[3] - 0.5 * (U[1:3] @ U[1:3]) / U[0])
    return torch.abs((U[1:3] @ n) / U[0]) + torch.sqrt(GAMMA * pr / U[0])


def _rusanov(UL, UR, n):
    aL, aR = _speed(UL, n), _speed(UR, n)
    return 0.5 * (_flux(UL, n) + _flux(UR, n)) - 0.5 * torch.where(aL >= aR, aL, aR) * (UR - UL)


def _mirror(U, n):
    return torch.cat([U[:1], U[1:3] - 2 * (U[1:3] @ n) * n, U[3:]])


def _points(f, *args):
    """f at every point (the leading dimensions of args), and its derivatives with respect to args[:-1]."""
    lead = args[0].shape[:-1]
    flat = [a.reshape(-1, a.shape[-1]) for a in args]
    v = torch.func.vmap(f)(*flat).reshape(*lead, 4)
    d = torch.func.vmap(torch.func.jacfwd(f, argnums=tuple(range(len(args) - 1))))(*flat)
    return v, [x.reshape(*lead, 4, 4) for x in d]


def _dense_system(c, X, u, cfl):
    """-R, dtau and the blocks of M/dtau + dR/du as a dict {"d", "e", "w", "n", "s"} of [n_r, n_theta, B, B]:
    the element itself and its neighbours at j+1, j-1, i+1, i-1."""
    p, n_theta, n_r = c["p"], c["n_theta"], c["n_r"]
    K, B = n_theta * n_r, _block(c)
    t, w = np.polynomial.legendre.leggauss(p + 2)
    V, D = _legendre(p, t)
    w = torch.as_tensor(w, device=DEV)
    one = _legendre(p, np.array([1.0, -1.0]))[0]

    def tensor2(eta, xi):  # psi_m(xi, eta), m = b (p+1) + a, points with xi fastest
        return torch.einsum("yb,xa->yxba", eta, xi).reshape(eta.shape[0] * xi.shape[0], -1)

    psi, pxi, peta = tensor2(V, V), tensor2(V, D), tensor2(D, V)
    W = torch.outer(w, w).reshape(-1)
    c0, c1, c2, c3 = (Y.reshape(K, 1, 2) for Y in (X[:-1], X[:-1].roll(-1, 1), X[1:].roll(-1, 1), X[1:]))
    tt = torch.as_tensor(t, device=DEV)
    xi, eta = tt.repeat(p + 2)[None, :, None], tt.repeat_interleave(p + 2)[None, :, None]
    dxi = 0.25 * ((1 - eta) * (c1 - c0) + (1 + eta) * (c2 - c3))
    deta = 0.25 * ((1 - xi) * (c3 - c0) + (1 + xi) * (c2 - c1))
    det = dxi[..., 0] * deta[..., 1] - deta[..., 0] * dxi[..., 1]
    grad = [W[None, :, None] * (deta[..., 1, None] * pxi - dxi[..., 1, None] * peta),
            W[None, :, None] * (dxi[..., 0, None] * peta - deta[..., 0, None] * pxi)]
    U = psi @ u                                                                       # [K, q^2, 4]
    pr = (GAMMA - 1) * (U[..., 3] - 0.5 * (U[..., 1] ** 2 + U[..., 2] ** 2) / U[..., 0])
    top = ((U[..., 1] ** 2 + U[..., 2] ** 2).sqrt() / U[..., 0] + (GAMMA * pr / U[..., 0]).sqrt()).amax(1)
    around = sum((b - a).norm(dim=-1) for a, b in ((c0, c1), (c1, c2), (c2, c3), (c3, c0)))[:, 0]
    dtau = float((cfl * (det @ W) / (top * (2 * p + 1) * around)).min())
    R = torch.zeros_like(u)
    d = torch.einsum("kq,qi,qj,vw->kivjw", det * W, psi, psi, torch.eye(4, dtype=torch.float64, device=DEV) / dtau)
    d = d.reshape(K, B, B)
    for G, n in zip(grad, torch.eye(2, dtype=torch.float64, device=DEV)):
        F, (J,) = _points(_flux, U, n.expand(*U.shape[:2], 2))
        R -= torch.einsum("kqm,kqv->kmv", G, F)
        for k in range(0, K, 4096):
            GJ = torch.einsum("kqi,kqvw->kivwq", G[k:k + 4096], J[k:k + 4096])
            d[k:k + 4096] -= torch.einsum("kivwq,qj->kivjw", GJ, psi).reshape(-1, B, B)
    R, d = R.reshape(n_r, n_theta, *R.shape[1:]), d.reshape(n_r, n_theta, B, B)
    off = {k: torch.zeros((n_r, n_theta, B, B), dtype=torch.float64, device=DEV) for k in "ewns"}
    off["d"] = d
    uu = u.reshape(n_r, n_theta, *u.shape[1:])
    face = dict(e=tensor2(V, one[:1]), w=tensor2(V, one[1:]), n=tensor2(one[:1], V), s=tensor2(one[1:], V))

    def side(P, J, Q):
        J = torch.einsum("qi,rcqvw,qj->rcivjw", P, J, Q)
        return J.reshape(*J.shape[:2], B, B)

    def normal(edge, sign):
        n = sign * torch.stack([edge[..., 1], -edge[..., 0]], -1)
        ln = n.norm(dim=-1)
        hw = 0.5 * ln[..., None] * w
        return (n / ln[..., None])[..., None, :].expand(*hw.shape, 2), hw

    # faces at j+1 (all, periodic) and at i+1 (all but the outer ring)
    for near, far, edge, sign, last in (("e", "w", (X[1:] - X[:-1]).roll(-1, 1), 1.0, n_r),
                                        ("n", "s", (X.roll(-1, 1) - X)[1:-1], -1.0, n_r - 1)):
        if last == 0:
            continue
        n, hw = normal(edge, sign)
        ur = uu.roll(-1, 1) if near == "e" else uu[1:]
        F, (JL, JR) = _points(_rusanov, face[near] @ uu[:last], face[far] @ ur, n)
        F, JL, JR = F * hw[..., None], JL * hw[..., None, None], JR * hw[..., None, None]
        R[:last] += torch.einsum("qm,rcqv->rcmv", face[near], F)
        back = torch.einsum("qm,rcqv->rcmv", face[far], F)
        own = side(face[far], JR, face[far])
        d[:last] += side(face[near], JL, face[near])
        off[near][:last] = side(face[near], JR, face[far])
        if near == "e":
            R -= back.roll(1, 1)
            d -= own.roll(1, 1)
            off[far] -= side(face[far], JL, face[near]).roll(1, 1)
        else:
            R[1:] -= back
            d[1:] -= own
            off[far][1:] -= side(face[far], JL, face[near])
    al = math.radians(2.0)
    vel = c["mach"] * torch.tensor([math.cos(al), math.sin(al)], dtype=torch.float64, device=DEV)
    free = torch.cat([torch.ones(1, dtype=torch.float64, device=DEV), vel,
                      (1 / GAMMA / (GAMMA - 1) + 0.5 * vel @ vel)[None]])
    wall = c.get("bc", "wall") == "wall"
    for i, name, edge, sign in ((0, "s", X[0].roll(-1, 0) - X[0], 1.0), (n_r - 1, "n", X[-1].roll(-1, 0) - X[-1], -1.0)):
        n, hw = normal(edge[None], sign)
        if name == "s" and wall:
            F, (J,) = _points(lambda a, m: _rusanov(a, _mirror(a, m), m), face[name] @ uu[i:i + 1], n)
        else:
            F, (J,) = _points(lambda a, m: _rusanov(a, free, m), face[name] @ uu[i:i + 1], n)
        R[i:i + 1] += torch.einsum("qm,rcqv->rcmv", face[name], F * hw[..., None])
        d[i:i + 1] += side(face[name], J * hw[..., None, None], face[name])
    return -R.reshape(-1), off, dtau


def _order(n_theta, n_r):
    """For each stored block, ascending columns in a row: its place in the five [n_r, n_theta] block arrays."""
    e = np.arange(n_theta * n_r)
    i, j = e // n_theta, e % n_theta
    cols = np.stack([e, i * n_theta + (j + 1) % n_theta, i * n_theta + (j - 1) % n_theta,
                     np.where(i < n_r - 1, e + n_theta, -1), np.where(i > 0, e - n_theta, -1)], 1)
    at = np.argsort(cols, 1, kind="stable")
    cols = np.take_along_axis(cols, at, 1)
    place = at * len(e) + e[:, None]
    return torch.as_tensor(place[cols >= 0], device=DEV)


def _values(off, n_theta, n_r):
    every = torch.cat([off[k].reshape(n_theta * n_r, *off[k].shape[2:]) for k in "dewns"])
    return every[_order(n_theta, n_r)].transpose(1, 2).reshape(-1)


def _product(off, x, transpose=False):
    n_r, n_theta, B = off["d"].shape[:3]
    x = x.reshape(n_r, n_theta, B, 1)
    if not transpose:
        y = off["d"] @ x + off["e"] @ x.roll(-1, 1) + off["w"] @ x.roll(1, 1)
        y[:-1] += off["n"][:-1] @ x[1:]
        y[1:] += off["s"][1:] @ x[:-1]
    else:
        t = {k: v.transpose(2, 3) for k, v in off.items()}
        y = t["d"] @ x + (t["e"] @ x).roll(1, 1) + (t["w"] @ x).roll(-1, 1)
        y[1:] += t["n"][:-1] @ x[:-1]
        y[:-1] += t["s"][1:] @ x[1:]
    return y.reshape(-1)


def _solve_flops(c):
    return 5 * c["n_r"] * float(c["n_theta"] * _block(c)) ** 3


def _solve(off, b, transpose=False):
    """A x = b (or A^T x = b) by block elimination ring by ring in 64 bits, refined twice."""
    n_r, n_theta, B = off["d"].shape[:3]
    m = n_theta * B
    j = torch.arange(n_theta, device=DEV)

    def ring(i, kind):
        """The dense coupling of ring i with itself ("d"), the ring outside it ("n") or inside it ("s")."""
        M = torch.zeros((n_theta, n_theta, B, B), dtype=torch.float64, device=DEV)
        if not 0 <= i < n_r:
            return None
        M[j, j] = off[kind][i]
        if kind == "d":
            M[j, (j + 1) % n_theta] += off["e"][i]
            M[j, (j - 1) % n_theta] += off["w"][i]
        M = M.permute(0, 2, 1, 3).reshape(m, m)
        return M

    factors, ups = [], []
    for i in range(n_r):
        M = ring(i, "d")
        M = M.T if transpose else M
        if i:
            low = ring(i - 1, "n").T if transpose else ring(i, "s")
            M = M - low @ ups[-1]
        LU = torch.linalg.lu_factor(M.contiguous())
        factors.append(LU)
        if i < n_r - 1:
            up = ring(i + 1, "s").T if transpose else ring(i, "n")
            ups.append(torch.linalg.lu_solve(*LU, up.contiguous()))

    def once(r):
        r = r.reshape(n_r, m, 1)
        y = []
        for i in range(n_r):
            t = r[i]
            if i:
                z = y[-1].reshape(n_theta, B, 1)
                z = off["n"][i - 1].transpose(1, 2) @ z if transpose else off["s"][i] @ z
                t = t - z.reshape(m, 1)
            y.append(torch.linalg.lu_solve(*factors[i], t))
        for i in reversed(range(n_r - 1)):
            y[i] = y[i] - ups[i] @ y[i + 1]
        return torch.cat(y).reshape(-1)

    x = once(b)
    for _ in range(2):
        x = x + once(b - _product(off, x, transpose))
    return x


MOST_FLOPS = 1.1e13  # about ten seconds of dense 64-bit work


def _exact_march(c, X, u):
    res, cfls, dts, cfl = [], [], [], c["cfl"]
    for n in range(c["steps"] + 1):
        b, off, dtau = _dense_system(c, X, u, cfl)
        res.append(float(b.norm()))
        cfls.append(cfl)
        dts.append(dtau)
        if n < c["steps"]:
            u = u + _solve(off, b).reshape(u.shape)
            cfl = min(c["cfl"] * res[0] / res[-1], 1e6)
    return [u, np.array(res), np.array(cfls), np.array(dts)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "batched":
        out = []
        for q, c in enumerate(_systems(case)):
            if _solve_flops(c) > MOST_FLOPS / 4:
                out.append(None)
                continue
            b, off, _ = _dense_system(c, *_inputs(c, 1000 * seed + q), c["cfl"])
            out.append(_solve(off, b))
        return out if any(x is not None for x in out) else None
    solves = {"spmv": 0, "assemble": 0, "march": case.get("steps"), "adjoint": 2, "apply": 2}.get(kind, 1)
    if solves * _solve_flops(case) > MOST_FLOPS or (kind == "apply" and case["eps"] > 0):
        return None
    X, u = _inputs(case, seed)
    if kind == "march":
        return _exact_march(case, X, u)
    b, off, dtau = _dense_system(case, X, u, case["cfl"])
    v = _vector(b.numel(), seed)
    if kind == "assemble":
        return [b, _values(off, case["n_theta"], case["n_r"]), dtau]
    if kind == "spmv":
        return [_product(off, v), _product(off, v, True)]
    if kind == "apply":
        return [_solve(off, v), _solve(off, v, True)]
    if kind == "solve":
        return _solve(off, b, case["transpose"])
    x = _solve(off, b)
    if kind == "factor_solve":
        return x
    lam = _solve(off, v, True)
    n_theta, n_r, B = case["n_theta"], case["n_r"], _block(case)
    xr, lr = x.reshape(n_r, n_theta, 1, B), lam.reshape(n_r, n_theta, B, 1)
    grad = dict(d=-lr * xr, e=-lr * xr.roll(-1, 1), w=-lr * xr.roll(1, 1), n=-lr * xr.roll(-1, 0),
                s=-lr * xr.roll(1, 0))
    return [x, _values(grad, n_theta, n_r), lam]
