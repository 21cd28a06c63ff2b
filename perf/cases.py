"""What a user of the solver has it do, as cases that can be timed.

A case names a mesh (element counts, order, deformation amplitude), the call
that is made on it and its options; ``prepare`` sets the mesh up and makes
seeded data, ``run`` makes the call once through the public binding
(``paper_2504_10710_gb300.glls``), and ``exact`` gives the same result in plain
64-bit torch.  Kinds of call:

  solve    one Poisson problem from new right-hand-side and Dirichlet data on
           the device to the solution (one or several right-hand sides)
  batch    independent 2-D problems of uneven size in one work-list launch
  serve    requests on registered meshes through the request loop, host data
  cycle    one gamma-cycle, z = M^-1 r, for a caller's own outer iteration
  smooth   one damped line-smoothing step per axis on the finest level
  transfer the residual's restriction and a correction's prolongation
  apply    the operator on the finest level
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2504_10710_gb300 import glls

TOL = 1e-10


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------
def _solve(nelem, order, amp, precision, nrhs=1, gamma=1, summation="atomic", smoother="gll"):
    nz = nelem[2] if len(nelem) == 3 else 0
    return dict(kind="solve", nx=nelem[0], ny=nelem[1], nz=nz, order=order, amp=amp, precision=precision, nrhs=nrhs,
                gamma=gamma, summation=summation, smoother=smoother)


def _level(kind, nelem, order, amp, dtype, **more):
    nz = nelem[2] if len(nelem) == 3 else 0
    return dict(kind=kind, nx=nelem[0], ny=nelem[1], nz=nz, order=order, amp=amp, dtype=dtype, **more)


def listed():
    return [
        # the smallest problem that is solved in earnest: latency of one call
        dict(_solve((4, 4), 4, 0.0, "fp64"), name="solve2d_4x4_p4_fp64"),
        # the headline workload, in both precisions
        dict(_solve((64, 64), 8, 0.1, "mixed"), name="solve2d_64x64_p8_mixed"),
        dict(_solve((64, 64), 8, 0.1, "fp64"), name="solve2d_64x64_p8_fp64"),
        # a ragged grid of a high, odd order whose answer has to be the same bits on each run
        dict(_solve((45, 28), 11, 0.15, "mixed", summation="colored"), name="solve2d_45x28_p11_colored"),
        # the 3-D workload: one right-hand side, and its 32 together
        dict(_solve((16, 16, 16), 7, 0.15, "mixed"), name="solve3d_16_p7_mixed"),
        dict(_solve((16, 16, 16), 7, 0.15, "mixed", nrhs=32), name="solve3d_16_p7_mixed_32rhs"),
        # a ragged 3-D grid wholly in 64 bits
        dict(_solve((9, 13, 11), 5, 0.15, "fp64"), name="solve3d_9x13x11_p5_fp64"),
        # independent problems of uneven size and order, n in 4..64 and p in 4..12
        dict(kind="batch", count=24, meshes=3, name="batch2d_uneven_24"),
        # a burst of requests on resident 2-D and 3-D meshes, from and to host memory
        dict(kind="serve", requests=18, meshes=4, name="serve_burst_18"),
        # the preconditioner alone, for a caller's own Krylov method
        dict(_level("cycle", (64, 64), 8, 0.1, "f32", gamma=1), name="cycle2d_64x64_p8_f32"),
        # single steps on a large grid, far above the L2 cache
        dict(_level("smooth", (24, 24, 24), 8, 0.15, "f32"), name="smooth3d_24_p8_f32"),
        dict(_level("transfer", (20, 20, 20), 6, 0.15, "f32"), name="transfer3d_20_p6_f32"),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def _grid(rng, dim, cap):
    """Element counts and an order of the ranges the workloads span, at most `cap` nodes."""
    while True:
        if dim == 2:
            p = rng.randint(4, 12) if rng.random() < 0.85 else rng.randint(2, 16)
            ne = [_log_int(rng, 2, 64)] * 2 if rng.random() < 0.3 else [_log_int(rng, 2, 64) for _ in range(2)]
        else:
            p = rng.randint(4, 8) if rng.random() < 0.8 else rng.randint(2, 8)
            ne = [_log_int(rng, 3, 24)] * 3 if rng.random() < 0.3 else [_log_int(rng, 3, 24) for _ in range(3)]
        if math.prod(e * p + 1 for e in ne) <= cap:
            return ne, p


def draw(rng):
    u = rng.random()
    dim = 2 if rng.random() < 0.55 else 3
    amp = round(rng.uniform(0.0, 0.2 if dim == 2 else 0.15), 3)
    if u < 0.56:
        ne, p = _grid(rng, dim, 1_500_000)
        nrhs = rng.choice([1, 1, 1, 1, 2, 5, 8, 32])
        while nrhs > 1 and nrhs * math.prod(e * p + 1 for e in ne) > 20_000_000:
            nrhs //= 2
        return _solve(ne, p, amp, rng.choice(["mixed", "mixed", "fp64"]), nrhs=nrhs, gamma=rng.choice([1, 1, 1, 2]),
                      summation=rng.choice(["atomic"] * 5 + ["colored"]),
                      smoother=rng.choice(["gll"] * 6 + ["fem"]) if dim == 2 else "gll")
    if u < 0.64:
        return dict(kind="batch", count=_log_int(rng, 2, 24), meshes=rng.randrange(1 << 20))
    if u < 0.70:
        return dict(kind="serve", requests=_log_int(rng, 4, 18), meshes=rng.randrange(1 << 20))
    ne, p = _grid(rng, dim, 5_000_000)
    dtype = rng.choice(["f32", "f32", "f64"])
    if u < 0.80:
        ne, p = _grid(rng, dim, 1_500_000)
        return _level("cycle", ne, p, amp, dtype, gamma=rng.choice([1, 1, 2]))
    if u < 0.88:
        return _level("smooth", ne, p, amp, dtype)
    if u < 0.94:
        return _level("transfer", ne, p, amp, dtype)
    return _level("apply", ne, p, amp, dtype)


def _batch_meshes(case):
    rng = random.Random(case["meshes"])
    out = []
    for _ in range(case["count"]):
        n = rng.randint(4, 64)
        out.append(((n, n), rng.randint(4, 12), rng.uniform(0.0, 0.2)))
    return out


def _serve_meshes(case):
    """Two 2-D meshes and one 3-D mesh; the requests take them in turn."""
    rng = random.Random(case["meshes"])
    out = []
    for _ in range(2):
        n = rng.randint(4, 64)
        out.append(((n, n), rng.randint(4, 12), rng.uniform(0.0, 0.2)))
    n = rng.randint(8, 12)
    out.append(((n, n, n), rng.randint(4, 6), 0.15))
    return out


def _nelem(case):
    return (case["nx"], case["ny"]) + ((case["nz"],) if case["nz"] else ())


# --------------------------------------------------------------------------
# meshes and data
# --------------------------------------------------------------------------
def _gll_points(p):
    """Gauss-Lobatto-Legendre points: -1, 1 and the roots of L_p'."""
    if p == 1:
        return np.array([-1.0, 1.0])
    leg = np.polynomial.legendre.Legendre.basis(p)
    x = np.sort(leg.deriv().roots().real)
    for _ in range(3):                               # Newton on L_p'
        x = x - leg.deriv()(x) / leg.deriv(2)(x)
    return np.concatenate([[-1.0], x, [1.0]])


def _coords(nelem, p, amp):
    """Node coordinates [dim][...z][y][x] of the deformed unit square or cube."""
    t = (_gll_points(p) + 1.0) / 2.0
    lines = []
    for e in nelem:
        line = np.concatenate([(np.arange(e)[:, None] + t[None, :-1]).ravel(), [e]]) / e
        lines.append(line)
    grids = np.meshgrid(*lines[::-1], indexing="ij")[::-1]
    two_pi = 2.0 * np.pi
    if len(nelem) == 2:
        x, y = grids
        return np.stack([x, y + amp * np.sin(two_pi * x) * (1.0 - y)])
    x, y, z = grids
    return np.stack([x, y, z + amp * np.sin(two_pi * x) * np.cos(two_pi * y) * (1.0 - z)])


def _generator(seed, what):
    return np.random.default_rng([2504_10710, int(seed), what])


def _fourier(coords, rng, modes=16, kmax=8):
    """sum of `modes` products of sines of pi k x with N(0, 1) amplitudes."""
    sines = [[torch.sin((math.pi * k) * c) for k in range(1, kmax + 1)] for c in coords]
    a, ks = rng.standard_normal(modes), rng.integers(0, kmax, (modes, len(coords)))
    f = torch.zeros_like(coords[0])
    for m in range(modes):
        term = a[m] * sines[0][ks[m, 0]]
        for ax in range(1, len(coords)):
            term = term * sines[ax][ks[m, ax]]
        f += term
    return f


def _boundary_data(coords, rng, modes=4):
    g = torch.zeros_like(coords[0])
    for _ in range(modes):
        b, th = rng.standard_normal(), rng.uniform(0.0, 2 * math.pi)
        phase = th + sum(math.pi * int(c) * x for c, x in zip(rng.integers(0, 4, len(coords)), coords))
        g += b * torch.cos(phase)
    return g


def _data(nelem, p, amp, seed, nrhs=1, what=0):
    """(f of shape (nrhs, N), g of shape (N,)) on the device."""
    X = [torch.from_numpy(c).cuda() for c in _coords(nelem, p, amp)]
    f = torch.stack([_fourier(X, _generator(seed, 1000 * what + j)).reshape(-1) for j in range(nrhs)])
    return f, _boundary_data(X, _generator(seed, 1000 * what + 999)).reshape(-1)


def _problem(nelem, p, amp, nrhs=1, summation="atomic", smoother="gll"):
    return glls.Problem(len(nelem), nelem, p, _coords(nelem, p, amp), nrhs=nrhs,
                        summation=glls.SUM_COLORED if summation == "colored" else glls.SUM_ATOMIC,
                        smoother=glls.SMOOTHER_FEM if smoother == "fem" else glls.SMOOTHER_GLL)


def _interior_field(nelem, p, seed, what, dtype):
    """N(0, 1) nodal values, zero on the boundary, as the level calls want them."""
    shape = tuple(e * p + 1 for e in reversed(nelem))
    g = torch.Generator(device="cuda").manual_seed((int(seed) * 8 + what) & 0x7FFFFFFF)
    inner = tuple(slice(1, -1) for _ in shape)
    out = torch.zeros(shape, dtype=dtype, device="cuda")
    out[inner] = torch.randn(tuple(n - 2 for n in shape), generator=g, dtype=torch.float64, device="cuda").to(dtype)
    return out


def _opts(precision="mixed", gamma=1, smoother="gll"):
    return glls.opts(tol=TOL, max_iter=300, gamma=gamma, alpha=0.16 if smoother == "fem" else 2.0 / 3.0,
                     precision=glls.PREC_FP64 if precision == "fp64" else glls.PREC_MIXED)


def _torch_type(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


def prepare(case, seed):
    kind = case["kind"]
    if kind == "solve":
        ne, p = _nelem(case), case["order"]
        prob = _problem(ne, p, case["amp"], case["nrhs"], case["summation"], case["smoother"])
        f, g = _data(ne, p, case["amp"], seed, case["nrhs"])
        return dict(kind=kind, prob=prob, f=f, g=g, u=torch.empty_like(f),
                    opts=_opts(case["precision"], case["gamma"], case["smoother"]))
    if kind == "batch":
        probs, fs, gs = [], [], []
        for i, (ne, p, amp) in enumerate(_batch_meshes(case)):
            probs.append(_problem(ne, p, amp))
            f, g = _data(ne, p, amp, seed, what=i)
            fs.append(f[0])
            gs.append(g)
        return dict(kind=kind, probs=probs, f=fs, g=gs, u=[torch.empty_like(f) for f in fs], opts=_opts())
    if kind == "serve":
        server = glls.Server(64 << 30, slots=4)
        server.set_max_group(8)
        o, ids, gs, reqs = _opts(), [], [], []
        meshes = _serve_meshes(case)
        for i, (ne, p, amp) in enumerate(meshes):
            ids.append(server.register(len(ne), ne, p, _coords(ne, p, amp)))
            gs.append(_data(ne, p, amp, seed, 1, i)[1].cpu().numpy())
        for k in range(case["requests"]):
            i = k % len(meshes)
            ne, p, amp = meshes[i]
            f = _data(ne, p, amp, seed, 1, 10 + k)[0][0].cpu().numpy()
            reqs.append((ids[i], f, gs[i], np.zeros_like(f)))
        for mesh, f, g, u in reqs[: len(meshes)]:       # the meshes are resident before the burst
            server.poll(server.submit_mesh(mesh, f, g, o, u), wait=True)
        return dict(kind=kind, server=server, reqs=reqs, opts=o)
    ne, p, t = _nelem(case), case["order"], _torch_type(case)
    prob = _problem(ne, p, case["amp"])
    s = dict(kind=kind, prob=prob, level=prob.levels - 1, dim=prob.dim, r=_interior_field(ne, p, seed, 0, t))
    if kind == "cycle":
        s.update(z=torch.zeros_like(s["r"]), opts=_opts("mixed", case["gamma"]))
    else:
        s.update(x0=_interior_field(ne, p, seed, 1, t))
        s.update(x=s["x0"].clone())
    if kind == "transfer":
        pc = int(prob.info.order[prob.levels - 2])
        s.update(e=_interior_field(ne, pc, seed, 2, t))
        s.update(rc=torch.zeros_like(s["e"]))
    return s


def run(state):
    kind = state["kind"]
    if kind == "solve":
        prob = state["prob"]
        prob.set_rhs(state["f"])
        prob.set_dirichlet(state["g"])
        prob.solve(state["u"], state["opts"])
        return state["u"]
    if kind == "batch":
        for prob, f, g in zip(state["probs"], state["f"], state["g"]):
            prob.set_rhs(f)
            prob.set_dirichlet(g)
        glls.solve_batch(state["probs"], state["u"], state["opts"], worklist=True)
        return state["u"]
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit_mesh(mesh, f, g, state["opts"], u) for mesh, f, g, u in state["reqs"]]
        for t in tickets:
            server.poll(t, wait=True)
        return [u for _, _, _, u in state["reqs"]]
    prob, level = state["prob"], state["level"]
    if kind == "cycle":
        prob.precondition(state["opts"], state["r"], state["z"])
        return state["z"]
    if kind == "apply":
        prob.apply(level, state["x0"], state["x"])
        return state["x"]
    x = state["x"]
    x.copy_(state["x0"])
    if kind == "smooth":
        for axis in range(state["dim"]):
            prob.smooth(level, axis, 2.0 / 3.0, state["r"], x)
        return x
    prob.restrict(level, state["r"], x, state["rc"])
    prob.prolong_add(level, state["e"], x)
    return [state["rc"], x]


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------
def _chain(nelem, p):
    p0 = 1 if min(nelem) > 1 else 2
    out = [p]
    while out[-1] > p0:
        out.append(max(p0, out[-1] // 2))
    return out


def _sizes(nelem, p):
    """(nodes, element nodes, flops of one apply, values of the line operators)."""
    d, E = len(nelem), math.prod(nelem)
    nodes, local = math.prod(e * p + 1 for e in nelem), E * (p + 1) ** d
    flops = 4 * d * (p + 1) * local + (6 if d == 2 else 15) * local
    lines = sum(e * ((p - 1) * p // 2 + 2 * (p - 1) + 2) * math.prod(f * p - 1 for b, f in enumerate(nelem) if b != a)
                for a, e in enumerate(nelem)) if p > 1 else 0
    return nodes, local, flops, lines


def _mesh_work(nelem, p, size, nrhs=1, gamma=1):
    """(bytes of the operators of all levels, flops of one gamma-cycle)."""
    d = len(nelem)
    total = flops = 0
    for depth, q in enumerate(_chain(nelem, p)[:-1]):
        nodes, local, fl, lines = _sizes(nelem, q)
        total += size * (d * (d + 1) // 2 * local + lines)
        flops += gamma ** depth * (1 + gamma) * d * (fl + 2 * lines) * nrhs
    return total, flops


def _solve_work(nelem, p, precision="mixed", nrhs=1, gamma=1):
    iterations = 10 if len(nelem) == 2 else 14
    nodes, _, fl, _ = _sizes(nelem, p)
    total, flops = _mesh_work(nelem, p, 8 if precision == "fp64" else 4, nrhs, gamma)
    total += 8 * nodes * (2 * nrhs + 1)
    return total, iterations * (flops + nrhs * (fl + 12 * nodes))


def work(case):
    kind = case["kind"]
    if kind == "solve":
        parts = [_solve_work(_nelem(case), case["order"], case["precision"], case["nrhs"], case["gamma"])]
    elif kind == "batch":
        parts = [_solve_work(ne, p) for ne, p, _ in _batch_meshes(case)]
    elif kind == "serve":
        meshes = _serve_meshes(case)
        parts = [_solve_work(*meshes[k % len(meshes)][:2]) for k in range(case["requests"])]
    else:
        ne, p, size = _nelem(case), case["order"], 8 if case["dtype"] == "f64" else 4
        nodes, local, fl, lines = _sizes(ne, p)
        d = len(ne)
        G = d * (d + 1) // 2 * local
        if kind == "cycle":
            total, flops = _mesh_work(ne, p, size, 1, case["gamma"])
            parts = [(total + 2 * size * nodes, flops)]
        elif kind == "smooth":
            parts = [(size * (G + lines + 3 * nodes), d * fl + 2 * lines)]
        elif kind == "apply":
            parts = [(size * (G + 2 * nodes), fl)]
        else:
            coarse = _sizes(ne, _chain(ne, p)[1])[0]
            parts = [(size * (G + 3 * nodes + 2 * coarse), fl + 4 * d * (p + 1) * nodes)]
    return {"bytes": sum(b for b, _ in parts), "flops": sum(f for _, f in parts)}


# --------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# --------------------------------------------------------------------------
def _interp(x, y):
    """M[i, k] = l_k(y_i) for the Lagrange basis on the points x."""
    M = np.ones((len(y), len(x)))
    for k in range(len(x)):
        for m in range(len(x)):
            if m != k:
                M[:, k] *= (y - x[m]) / (x[k] - x[m])
    return M


def _derivative(x):
    w = np.array([1.0 / np.prod(np.delete(xk - x, k)) for k, xk in enumerate(x)])
    D = np.array([[0.0 if i == j else w[j] / w[i] / (x[i] - x[j]) for j in range(len(x))] for i in range(len(x))])
    D[np.diag_indices(len(x))] = -D.sum(axis=1)
    return D


def _along(M, t, axis):
    return torch.movedim(torch.tensordot(M, t, dims=([1], [axis])), 0, axis)


def _fold(t, ax_e, ax_l):
    """Sums the shared ends of neighbouring elements; the node axis is put last."""
    t = torch.movedim(t, (ax_e, ax_l), (-2, -1))
    E, n = t.shape[-2], t.shape[-1]
    out = torch.zeros(t.shape[:-2] + (E * (n - 1) + 1,), dtype=t.dtype, device=t.device)
    out[..., :-1] += t[..., :-1].reshape(t.shape[:-2] + (E * (n - 1),))
    out[..., n - 1::n - 1] += t[..., -1]
    return out


class _Grid:
    """One level of the discretisation: arrays [z][y][x], element arrays
    [Ez][Ey][Ex][k][j][i]; physical axis a is element axis d-1-a and local
    axis 2d-1-a."""

    def __init__(self, nelem, p, coords):
        self.d, self.nelem, self.p, self.coords = len(nelem), tuple(nelem), p, coords
        d = self.d
        x = _gll_points(p)
        lp = np.polynomial.legendre.Legendre.basis(p)(x)
        self.D = torch.from_numpy(_derivative(x)).cuda()
        rho = torch.from_numpy(2.0 / (p * (p + 1) * lp ** 2)).cuda()
        X = [self.elements(c) for c in coords]
        J = torch.stack([torch.stack([_along(self.D, X[b], 2 * d - 1 - a) for a in range(d)], -1) for b in range(d)], -2)
        det, inv = torch.linalg.det(J), torch.linalg.inv(J)
        w = torch.ones((1,) * (2 * d), dtype=torch.float64, device="cuda")
        for a in range(d):
            w = w * self.local(rho, a)
        self.G = [[w * det * (inv[..., a, :] * inv[..., b, :]).sum(-1) for b in range(d)] for a in range(d)]
        self.mass = self.assemble(w * det)

    def local(self, v, a):
        shape = [1] * (2 * self.d)
        shape[2 * self.d - 1 - a] = len(v)
        return v.reshape(shape)

    def elements(self, u):
        for ax in range(self.d):
            u = u.unfold(ax, self.p + 1, self.p)
        return u

    def assemble(self, t):
        for left in range(self.d, 0, -1):            # the slowest axis first; its nodes go to the end
            t = _fold(t, 0, left)
        return t

    def masked(self, u):
        out = torch.zeros_like(u)
        inner = tuple(slice(1, -1) for _ in range(self.d))
        out[inner] = u[inner]
        return out

    def apply_all(self, u):
        d = self.d
        ue = self.elements(u)
        g = [_along(self.D, ue, 2 * d - 1 - a) for a in range(d)]
        y = 0.0
        for a in range(d):
            y = y + _along(self.D.T, sum(self.G[a][b] * g[b] for b in range(d)), 2 * d - 1 - a)
        return self.assemble(y)

    def apply(self, u):
        return self.masked(self.apply_all(u))

    def diagonal(self):
        """Of A: the line matrices' diagonal."""
        d, D2, Dd = self.d, (self.D * self.D).T, torch.diagonal(self.D)
        t = 0.0
        for a in range(d):
            t = t + _along(D2, self.G[a][a], 2 * d - 1 - a)
            for b in range(d):
                if b != a:
                    t = t + self.G[a][b] * self.local(Dd, a) * self.local(Dd, b)
        return self.assemble(t)

    def solve(self, b, tol=1e-13):
        """Jacobi-preconditioned CG for A x = b, restarted on the true residual."""
        dia = self.diagonal()
        x, r = torch.zeros_like(b), b.clone()
        r0 = float(b.norm())
        if r0 == 0.0:
            return x
        for _ in range(3):
            z = self.masked(r / dia)
            q, rz, goal = z.clone(), (r * z).sum(), max(1e-8 * float(r.norm()), 0.1 * tol * r0)
            for it in range(20000):
                Aq = self.apply(q)
                al = rz / (q * Aq).sum()
                x += al * q
                r -= al * Aq
                if it % 20 == 19 and float(r.norm()) <= goal:
                    break
                z = self.masked(r / dia)
                new = (r * z).sum()
                q = z + (new / rz) * q
                rz = new
            r = self.masked(b - self.apply(x))
            if float(r.norm()) <= tol * r0:
                break
        return x

    def line_blocks(self, s):
        """The principal submatrices of A on the interior lines along axis s:
        [other axes, slowest first][n][n]."""
        d, p, D = self.d, self.p, self.D
        Dd, ls = torch.diagonal(D), 2 * d - 1 - s
        last = lambda t: torch.movedim(t, ls, -1)  # noqa: E731
        shape = self.G[0][0].shape
        K = torch.einsum("...q,qi,qj->...ij", last(self.G[s][s]), D, D)
        diag = torch.zeros(shape, dtype=torch.float64, device="cuda")
        others = [a for a in range(d) if a != s]
        for t in others:
            c = last(self.G[s][t] * self.local(Dd, t))               # at q_s = the column's node
            K = K + c[..., None, :] * D.T + c[..., :, None] * D
            diag += _along((D * D).T, self.G[t][t], 2 * d - 1 - t)
            for v in others:
                if v != t:
                    diag += self.G[t][v] * self.local(Dd, t) * self.local(Dd, v)
        K = K + torch.diag_embed(last(diag))
        K = torch.movedim(K, d - 1 - s, -3)          # the others' elements, the others' nodes, E_s, i, j
        for left in range(d - 1, 0, -1):
            K = _fold(K, 0, left)                    # E_s, i, j, the others' nodes
        K = torch.movedim(K, (0, 1, 2), (-3, -2, -1))
        E = self.nelem[s]
        K = K[tuple(slice(1, -1) for _ in others)]
        M = torch.zeros(K.shape[:-3] + (E * p + 1, E * p + 1), dtype=torch.float64, device="cuda")
        for e in range(E):
            M[..., e * p:(e + 1) * p + 1, e * p:(e + 1) * p + 1] += K[..., e, :, :]
        return M[..., 1:-1, 1:-1]

    def smooth(self, s, alpha, r, x):
        g = r - (self.apply(x) if x is not None else 0.0)
        inner = tuple(slice(1, -1) for _ in range(self.d))
        gl = torch.movedim(g[inner], self.d - 1 - s, -1)
        M = self.line_blocks(s)
        n = M.shape[-1]
        M, rhs = M.reshape(-1, n, n), gl.reshape(-1, n, 1)
        sol = torch.cat([torch.cholesky_solve(b, torch.linalg.cholesky(m))
                         for m, b in zip(M.split(4096), rhs.split(4096))]).reshape(gl.shape)
        out = torch.zeros_like(r) if x is None else x.clone()
        out[inner] += alpha * torch.movedim(sol, -1, self.d - 1 - s)
        return out


def _to_order(nelem, p_from, p_to):
    """Per axis, the 1-D interpolation from order p_from to the nodes of p_to."""
    J = _interp(_gll_points(p_from), _gll_points(p_to))
    out = []
    for E in nelem:
        M = np.zeros((E * p_to + 1, E * p_from + 1))
        for e in range(E):
            M[e * p_to:(e + 1) * p_to + 1, e * p_from:(e + 1) * p_from + 1] = J
        out.append(torch.from_numpy(M).cuda())
    return out


def _tensor_product(Ms, u, transpose=False):
    d = len(Ms)
    for a, M in enumerate(Ms):
        u = _along(M.T if transpose else M, u, d - 1 - a)
    return u


def _fine_grid(nelem, p, amp):
    return _Grid(nelem, p, [torch.from_numpy(c).cuda() for c in _coords(nelem, p, amp)])


def _gamma_cycle(nelem, p, amp, r, gamma, alpha):
    grids = [_fine_grid(nelem, p, amp)]
    for q in _chain(nelem, p)[1:]:
        up = _to_order(nelem, grids[-1].p, q)
        grids.append(_Grid(nelem, q, [_tensor_product(up, c) for c in grids[-1].coords]))

    def cycle(k, rk):
        g = grids[k]
        if k == len(grids) - 1:
            return g.solve(rk, 1e-14)
        P, x = _to_order(nelem, grids[k + 1].p, g.p), None
        for s in range(g.d):
            x = g.smooth(s, alpha, rk, x)
        for _ in range(gamma):
            rc = grids[k + 1].masked(_tensor_product(P, rk - g.apply(x), True))
            x = x + _tensor_product(P, cycle(k + 1, rc))
            for s in reversed(range(g.d)):
                x = g.smooth(s, alpha, rk, x)
        return x

    return cycle(0, r)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("batch", "serve"):
        return None
    ne, p, amp = _nelem(case), case["order"], case["amp"]
    if kind == "solve":
        if case["nrhs"] * math.prod(e * p + 1 for e in ne) > 2_000_000:
            return None
        f, g = _data(ne, p, amp, seed, case["nrhs"])
        grid = _fine_grid(ne, p, amp)
        shape = grid.mass.shape
        v = g.reshape(shape) - grid.masked(g.reshape(shape))
        out = []
        for fj in f:
            b = grid.masked(grid.mass * fj.reshape(shape) - grid.apply_all(v))
            out.append((grid.solve(b) + v).reshape(-1))
        return torch.stack(out)
    t = _torch_type(case)
    r = _interior_field(ne, p, seed, 0, t).double()
    if kind == "cycle":
        return _gamma_cycle(ne, p, amp, r, case["gamma"], 2.0 / 3.0)
    grid = _fine_grid(ne, p, amp)
    x = _interior_field(ne, p, seed, 1, t).double()
    if kind == "apply":
        return grid.apply(x)
    if kind == "smooth":
        alpha = 2.0 / 3.0
        for s in range(grid.d):
            x = grid.smooth(s, alpha, r, x)
        return x
    pc = _chain(ne, p)[1]
    P = _to_order(ne, pc, p)
    coarse_shape = tuple(e * pc + 1 for e in reversed(ne))
    inner = tuple(slice(1, -1) for _ in ne)
    rc = torch.zeros(coarse_shape, dtype=torch.float64, device="cuda")
    rc[inner] = _tensor_product(P, r - grid.apply(x), True)[inner]
    return [rc, x + _tensor_product(P, _interior_field(ne, pc, seed, 2, t).double())]
