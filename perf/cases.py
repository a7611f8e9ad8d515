"""Measured workloads: what users of this library have it do, through its Python entry points.

A case is a dict of plain values: a mesh (elements per axis, elements per subdomain, grading
of the tensor grid, Dirichlet faces), the solver's options and a kind of call:

  solve            one time step of a sequence, x = K^{-1} f (Solver.solve), deflated by the
                   basis recycled over the steps before it when k > 0
  gradient         one training step through PoissonSolve: forward solve, backward (adjoint) solve
                   and the gradients with respect to the load and the log-coefficient field
  ensemble         one time step of `members` sequences solved as one block (Solver.solve_batch)
  schur            y = A x on the interface (Solver.schur_apply), e.g. inside a user's own Krylov method
  schur_batch      the same for several vectors at once (Solver.schur_apply_batch)
  condense_recover static condensation of a load and back-substitution of interface values

A solver is set up once per matrix and kept, as a program that solves a sequence does; the loads,
targets and vectors are made on the device from the seed. A sequence's passes go back and forth over
a few neighbouring time steps, so that each is a step of the size a time loop makes.
"""
import math
from collections import OrderedDict
from types import SimpleNamespace

import numpy as np
import torch

import paper_2412_17543_gb300 as dd

X0, X1, Y0, Y1, Z0, Z1 = 1, 2, 4, 8, 16, 32  # Dirichlet face bits

WARM = 6     # steps of a recycled sequence before the measured ones (its basis is built meanwhile)
STEPS = 4    # neighbouring steps that the passes of a sequence go back and forth over
ENS_STEPS = 2

_BASE = dict(sx=8, sy=8, sz=8, grade=1.08, aspect=20.0, faces=X1, levels=3, group=4, edges=1, adaptive=0, mixed=1,
             flexible=1, coef=0, k=0, rtol=1e-9)


def _case(kind, n, **kw):
    nx, ny, nz = n if isinstance(n, tuple) else (n, n, n)
    return dict(_BASE, kind=kind, nx=nx, ny=ny, nz=nz, **kw)


def listed():
    return [
        # the smallest workload of the repository: uniform 16^3, 64 subdomains of 4^3, two levels, plain FP64 PCG;
        # a solve is a few dozen short launches
        dict(_case("solve", 16), name="solve 16^3 fp64", sx=4, sy=4, sz=4, grade=1.0, levels=2, edges=0, mixed=0,
             flexible=0, rtol=1e-8),
        # a ragged box with subdomains that are not cubes (30 x 24 x 20 elements in blocks of 6 x 4 x 5), Dirichlet data
        # on two faces: what a user's own domain looks like
        dict(_case("solve", (30, 24, 20), k=8), name="solve 30x24x20 mixed", sx=6, sy=4, sz=5, faces=X0 | X1, group=2),
        # the plain FP64 arm (options at their defaults) at a middle size
        dict(_case("solve", 48), name="solve 48^3 fp64", mixed=0, flexible=0, group=2),
        # pure Neumann data (no Dirichlet face), mixed precision
        dict(_case("solve", 40, k=8), name="solve 40^3 neumann", faces=0, group=2),
        # one step of the repository's 64^3 sequence: three levels, basis of 20 columns, mixed precision
        dict(_case("solve", 64, k=20), name="solve 64^3 mixed", rtol=1e-8),
        # one step of the benchmark's 128^3 sequence: 4096 subdomains, adaptive constraints, basis of 40 columns
        dict(_case("solve", 128, k=40), name="solve 128^3 mixed", aspect=40.0, adaptive=1, rtol=1e-8),
        # one training step of the differentiation workload: 64^3, k = exp(g) varying from element to element
        dict(_case("gradient", 64, k=20), name="gradient 64^3", coef=1, rtol=1e-10),
        # one block step of the repository's ensemble of 32 sequences on 96^3
        dict(_case("ensemble", 96, k=40, members=32), name="ensemble 96^3 x32", aspect=40.0, rtol=1e-8),
        # a small ensemble that does not fill the block, on a box
        dict(_case("ensemble", (48, 32, 40), k=8, members=12), name="ensemble 48x32x40 x12", group=2),
        # operators alone, as a user's own iteration calls them
        dict(_case("schur", 64), name="schur 64^3 df64"),
        dict(_case("schur_batch", (72, 48, 40), members=24), name="schur 72x48x40 x24", group=2),
        # condensation and back-substitution on the 96^3 mesh in FP64
        dict(_case("condense_recover", 96), name="condense+recover 96^3", aspect=40.0, mixed=0, flexible=0),
    ]


def draw(rng):
    """One more case: sizes spread over their logarithm between the listed ones, every kind of call."""
    kind = rng.choice(["solve", "solve", "solve", "solve", "ensemble", "ensemble", "gradient", "schur", "schur_batch",
                       "condense_recover"])
    s = [rng.choice([4, 5, 6, 8, 8, 8])] * 3
    if rng.random() < 0.25:
        s = [rng.choice([3, 4, 5, 6, 7, 8]) for _ in range(3)]
    most = {"ensemble": 7, "gradient": 6}.get(kind, 12)
    b = [max(2, int(round(math.exp(rng.uniform(math.log(2), math.log(most)))))) for _ in range(3)]
    blocks = b[0] * b[1] * b[2]
    c = _case(kind, (s[0] * b[0], s[1] * b[1], s[2] * b[2]))
    c.update(sx=s[0], sy=s[1], sz=s[2], faces=rng.choice([X1, X1, X0 | X1, X1 | Y0 | Z1]),
             grade=rng.choice([1.0, 1.08, 1.08, 1.3]), aspect=rng.choice([20.0, 40.0]))
    c.update(levels=2 if blocks <= 40 else 3, group=2 if max(b) <= 5 else 4)
    if c["levels"] == 3 and c["group"] == 4 and max(b) <= 4:
        c["group"] = 2
    fp64 = rng.random() < 0.25
    c.update(mixed=0 if fp64 else 1, flexible=0 if fp64 else 1)
    if kind in ("solve", "gradient"):
        c["k"] = rng.choice([0, 8, 20])
    if kind == "gradient":
        c.update(coef=1, rtol=1e-10)
    if kind == "ensemble":
        c.update(k=rng.choice([0, 8, 20]), members=rng.randint(3, 32))
    if kind == "schur_batch":
        c["members"] = rng.randint(3, 32)
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _coords(n, ratio, aspect):
    """n elements of [0, 1] graded towards the middle, largest to smallest at most `aspect`."""
    if ratio == 1.0 or n < 4:
        return np.linspace(0.0, 1.0, n + 1)
    r = min(ratio, aspect ** (1.0 / (n / 2 - 1)))
    h = r ** (np.abs(np.arange(n) - (n - 1) / 2.0) - 0.5)
    x = np.concatenate([[0.0], np.cumsum(h / h.sum())])
    x[-1] = 1.0
    return x


def _axes(c):
    """Per axis: node coordinates, first and past-the-last free node."""
    lo, hi = (X0, Y0, Z0), (X1, Y1, Z1)
    out = []
    for a, n in enumerate((c["nx"], c["ny"], c["nz"])):
        out.append((_coords(n, c["grade"], c["aspect"]), 1 if c["faces"] & lo[a] else 0, n if c["faces"] & hi[a] else n + 1))
    return out


def _field(c):
    """The log-coefficient field g per element [nz][ny][nx]: a smooth random field of the matrix, not of the inputs."""
    rng = np.random.default_rng(40)
    grids = [0.5 * (x[1:] + x[:-1]) for x, _, _ in _axes(c)]
    g = np.zeros((c["nz"], c["ny"], c["nx"]))
    for _ in range(24):
        w, p = rng.normal(0.0, 10.0, 3), rng.uniform(0.0, 2 * math.pi)
        gx, gy, gz = (w[a] * grids[a] for a in range(3))
        g += np.cos(gz[:, None, None] + gy[None, :, None] + gx[None, None, :] + p)
    return np.ascontiguousarray(g / g.std())


_solvers = OrderedDict()  # the matrices in use: a program keeps a solver for as long as it solves with its matrix
_INPUT_ONLY = ("kind", "name", "k", "rtol", "members")


def _solver(c):
    key = tuple(sorted((k, v) for k, v in c.items() if k not in _INPUT_ONLY))
    if key not in _solvers:
        (x, _, _), (y, _, _), (z, _, _) = _axes(c)
        mesh = SimpleNamespace(nx=c["nx"], ny=c["ny"], nz=c["nz"], xc=x, yc=y, zc=z, sub=(c["sx"], c["sy"], c["sz"]),
                               dirichlet=c["faces"], coef=np.exp(_field(c)) if c["coef"] else None)
        _solvers[key] = dd.Solver(mesh, levels=c["levels"], coarse_group=c["group"], use_corners=1, use_edges=c["edges"],
                                  use_faces=1, weights="diag", adaptive=c["adaptive"], tau=10.0,
                                  schur_prec="df64" if c["mixed"] else "fp64",
                                  precond_prec="fp32" if c["mixed"] else "fp64", flexible=c["flexible"])
        while len(_solvers) > 2:
            _solvers.popitem(last=False)
    _solvers.move_to_end(key)
    return _solvers[key]


def _gen(*seed):
    h = 0
    for v in seed:
        h = (h * 1000003 + int(v) + 12345) % (1 << 61)
    return torch.Generator(device="cuda").manual_seed(h)


def _loads(c, seed, member, steps):
    """[steps][n_free] load vectors: eight advected Gaussian bumps and white noise times the nodal volumes."""
    dev = torch.device("cuda")
    ax, vol = [], []
    for x, a, b in _axes(c):
        h = np.diff(x)
        v = np.zeros(len(x))
        v[:-1] += 0.5 * h
        v[1:] += 0.5 * h
        ax.append(torch.tensor(x[a:b], device=dev))
        vol.append(torch.tensor(v[a:b], device=dev))
    r = np.random.default_rng([seed % (1 << 31), member])
    amp = torch.tensor(r.standard_normal(8), device=dev)
    w = torch.tensor(r.uniform(0.05, 0.2, 8), device=dev)
    c0, v0 = r.uniform(0.0, 1.0, (8, 3)), r.standard_normal((8, 3))
    v0 *= 0.5 / np.linalg.norm(v0, axis=1, keepdims=True)
    out = torch.empty(steps, ax[0].numel() * ax[1].numel() * ax[2].numel(), dtype=torch.float64, device=dev)
    g = _gen(seed, member, 1)
    for t in range(steps):
        cen = torch.tensor(np.mod(c0 + v0 * (0.05 * t), 1.0), device=dev)
        e = [torch.exp(-((ax[a][None, :] - cen[:, a, None]) ** 2) / (2.0 * w[:, None] ** 2)) * vol[a] for a in range(3)]
        f = torch.einsum("mz,my,mx->zyx", amp[:, None] * e[2], e[1], e[0]).reshape(-1)
        xi = torch.randn(f.numel(), dtype=torch.float64, device=dev, generator=g)
        out[t] = f + 1e-3 * xi * (vol[2][:, None, None] * vol[1][None, :, None] * vol[0][None, None, :]).reshape(-1)
    return out


def _warm(c):
    return WARM if c["k"] else 1


def _back_and_forth(n):
    """0, 1, ..., n - 1, n - 2, ..., 1, 0, 1, ..."""
    i, d = 0, 1
    while True:
        yield i
        if n > 1:
            if not 0 <= i + d < n:
                d = -d
            i += d


def _n_free(c):
    return math.prod(b - a for _, a, b in _axes(c))


def _target(c, seed, x_rms):
    return x_rms * torch.randn(_n_free(c), dtype=torch.float64, device="cuda", generator=_gen(seed, 2))


def _interface_input(c, seed, rows):
    m = _cut(c).sum()
    return torch.randn(rows, int(m), dtype=torch.float64, device="cuda", generator=_gen(seed, 3))


def prepare(case, seed):
    c = case
    S = _solver(c)
    kind = c["kind"]
    if kind == "solve":
        rec = S.recycler(c["k"])
        W = _warm(c)
        F = _loads(c, seed, 0, W + STEPS)
        for t in range(W):
            S.solve(F[t], rec, rtol=c["rtol"])
        return dict(c=c, S=S, rec=rec, F=F[W:].contiguous(), order=_back_and_forth(STEPS))
    if kind == "ensemble":
        rec = S.ensemble_recycler(c["k"])
        W = _warm(c)
        F = torch.stack([_loads(c, seed, j, W + ENS_STEPS) for j in range(c["members"])], dim=1)
        for t in range(W):
            S.solve_batch(F[t], rec, rtol=c["rtol"])
        return dict(c=c, S=S, rec=rec, F=F[W:].clone(), order=_back_and_forth(ENS_STEPS))
    if kind == "gradient":
        rec = S.recycler(c["k"])
        W = _warm(c)
        F = _loads(c, seed, 0, W + STEPS)
        for t in range(W):
            x, _ = S.solve(F[t], rec, rtol=c["rtol"])
        f = [F[W + t].clone().requires_grad_() for t in range(STEPS)]
        g = torch.tensor(_field(c), device="cuda").requires_grad_()
        return dict(c=c, S=S, rec=rec, f=f, g=g, target=_target(c, seed, 1e-2), order=_back_and_forth(STEPS))
    if kind == "schur":
        return dict(c=c, S=S, x=_interface_input(c, seed, 1)[0])
    if kind == "schur_batch":
        return dict(c=c, S=S, x=_interface_input(c, seed, c["members"]))
    return dict(c=c, S=S, f=_loads(c, seed, 0, 1)[0], xg=_interface_input(c, seed, 1)[0])


def run(state):
    c, S = state["c"], state["S"]
    kind = c["kind"]
    if kind == "solve":
        x, _ = S.solve(state["F"][next(state["order"])], state["rec"], rtol=c["rtol"])
        return x
    if kind == "ensemble":
        x, _ = S.solve_batch(state["F"][next(state["order"])], state["rec"], rtol=c["rtol"])
        return x
    if kind == "gradient":
        f, g = state["f"][next(state["order"])], state["g"]
        f.grad = g.grad = None
        x = dd.PoissonSolve.apply(f, g, S, state["rec"], c["rtol"], c["rtol"])
        loss = 0.5 * (x - state["target"]).square().sum()
        loss.backward()
        return {"x": x.detach(), "grad_f": f.grad, "grad_g": g.grad}
    if kind == "schur":
        return S.schur_apply(state["x"])
    if kind == "schur_batch":
        return S.schur_apply_batch(state["x"])
    return [S.condense(state["f"]), S.recover(state["f"], state["xg"])]


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    c = case
    counts = []  # per axis and block: (interior nodes, all free nodes)
    for (x, a, b), s in zip(_axes(c), (c["sx"], c["sy"], c["sz"])):
        n = len(x) - 1
        counts.append([(sum(1 for p in range(j, j + s + 1) if a <= p < b and (p % s or p in (0, n))),
                        sum(1 for p in range(j, j + s + 1) if a <= p < b)) for j in range(0, n, s)])
    n_free, n_gamma = _n_free(c), int(_cut(c).sum())
    tri = kii = flat = 0.0
    for iz, az in counts[2]:
        for iy, ay in counts[1]:
            for ix, ax in counts[0]:
                i, g = ix * iy * iz, ax * ay * az - ix * iy * iz
                tri += g * (g + 1) / 2
                kii += i * (i + 1) / 2 if c["coef"] else i + 2 * i * (ix + iy + iz)
                flat += g
    m = c.get("members", 1)
    # one Schur application: every vector once, K_II^{-1} (packed triangles for a varying coefficient, else the
    # inverse eigenvalue sums), 27 products per interface copy
    schur_b = 8.0 * (2 * n_gamma * m + flat + (kii if c["coef"] else n_free - n_gamma))
    schur_f = m * (2.0 * 2 * kii + 2.0 * 27 * flat)
    if c["kind"] == "schur" or c["kind"] == "schur_batch":
        return {"bytes": schur_b, "flops": schur_f}
    if c["kind"] == "condense_recover":
        return {"bytes": 8.0 * (3 * n_free + 2 * n_gamma), "flops": 2 * schur_f}
    # one PCG iteration: a Schur application, the local operators N_i once, the basis once in each direction
    its = 8 + 0.004 * max(c["nx"], c["ny"], c["nz"]) ** 2
    solves = 2 if c["kind"] == "gradient" else 1
    eb = 4.0 if c["mixed"] else 8.0
    it_b = schur_b + eb * tri + 8.0 * 4 * n_gamma * m + c["k"] * n_gamma * (8.0 + eb)
    it_f = schur_f + m * (4.0 * tri + 4.0 * c["k"] * n_gamma)
    return {"bytes": solves * (16.0 * n_free * m + its * it_b), "flops": solves * its * it_f}


# ---------------------------------------------------------------------------
# the same results from plain torch in FP64
# ---------------------------------------------------------------------------
def _cut(c):
    """Free nodes [z][y][x] on a plane between subdomains (nodes of more than one subdomain)."""
    on = []
    for (x, a, b), s in zip(_axes(c), (c["sx"], c["sy"], c["sz"])):
        p = np.arange(a, b)
        on.append((p % s == 0) & (p > 0) & (p < len(x) - 1))
    return on[2][:, None, None] | on[1][None, :, None] | on[0][None, None, :]


def _axis_matrices(c):
    """Per axis the stiffness and mass matrices of linear elements on the free nodes."""
    out = []
    for x, a, b in _axes(c):
        h, n = np.diff(x), len(x)
        K, M = np.zeros((n, n)), np.zeros((n, n))
        for e, v in enumerate(h):
            K[e:e + 2, e:e + 2] += np.array([[1.0, -1.0], [-1.0, 1.0]]) / v
            M[e:e + 2, e:e + 2] += np.array([[2.0, 1.0], [1.0, 2.0]]) * (v / 6)
        out.append((K[a:b, a:b], M[a:b, a:b]))
    return out


def _along(A, v, axis):
    """A applied along `axis` (0 x, 1 y, 2 z) of v[..., z, y, x]."""
    d = v.dim() - 1 - axis
    return torch.movedim(torch.tensordot(A, v, dims=([1], [d])), 0, d)


def _apply(KM, v):
    """K v for a coefficient of one: the sum of the three products of axis matrices."""
    (Kx, Mx), (Ky, My), (Kz, Mz) = KM
    a, b = _along(Kx, v, 0), _along(Mx, v, 0)
    t = _along(My, a, 1) + _along(Ky, b, 1)
    return _along(Mz, t, 2) + _along(Kz, _along(My, b, 1), 2)


def _tensors(mats):
    return [tuple(torch.tensor(np.ascontiguousarray(m), device="cuda") for m in km) for km in mats]


def _inverse(mats):
    """v -> K^{-1} v on the tensor set of the given axis matrices, by their generalized eigenvectors (a zero
    eigenvalue sum, the constants, is left out), with one step of refinement."""
    V, lam = [], []
    for K, M in mats:
        L = np.linalg.cholesky(M)
        Li = np.linalg.inv(L)
        C = Li @ K @ Li.T
        w, U = np.linalg.eigh(0.5 * (C + C.T))
        V.append(torch.tensor(Li.T @ U, device="cuda"))
        lam.append(torch.tensor(w, device="cuda"))
    D = lam[2][:, None, None] + lam[1][None, :, None] + lam[0][None, None, :]
    D = torch.where(D > 1e-10 * D.max(), 1.0 / D, torch.zeros_like(D))
    KM = _tensors(mats)

    def once(v):
        for a in range(3):
            v = _along(V[a].T.contiguous(), v, a)
        v = v * D
        for a in range(3):
            v = _along(V[a], v, a)
        return v

    def solve(v):
        x = once(v)
        return x + once(v - _apply(KM, x))
    return solve


def _interior(c, mats):
    """The axis matrices on the nodes off the cut planes (the interior nodes are the tensor set of these)."""
    out, keep = [], []
    for (K, M), (x, a, b), s in zip(mats, _axes(c), (c["sx"], c["sy"], c["sz"])):
        p = np.arange(a, b)
        i = np.nonzero((p % s != 0) | (p == 0) | (p == len(x) - 1))[0]
        out.append((K[np.ix_(i, i)], M[np.ix_(i, i)]))
        keep.append(torch.tensor(i, device="cuda"))
    return out, keep


class _Elements:
    """K(k) v and the element energies for a coefficient per element, brick by brick."""

    def __init__(self, c):
        self.box = [(a, b, len(x)) for x, a, b in _axes(c)]
        h = [torch.tensor(np.diff(x), device="cuda") for x, _, _ in _axes(c)]
        hx, hy, hz = h[0][None, None, :], h[1][None, :, None], h[2][:, None, None]
        f = (hy * hz / (36 * hx), hx * hz / (36 * hy), hx * hy / (36 * hz))
        self.kd = []  # entry of two corners that differ along the axes in d
        for d in range(8):
            s = [-1.0 if d >> a & 1 else 1.0 for a in range(3)]
            m = [1.0 if d >> a & 1 else 2.0 for a in range(3)]
            self.kd.append(f[0] * (s[0] * m[1] * m[2]) + f[1] * (m[0] * s[1] * m[2]) + f[2] * (m[0] * m[1] * s[2]))
        self.k = torch.tensor(np.exp(_field(c)), device="cuda")

    def grid(self, v):
        (xa, xb, nx), (ya, yb, ny), (za, zb, nz) = self.box
        g = torch.zeros(nz, ny, nx, dtype=torch.float64, device="cuda")
        g[za:zb, ya:yb, xa:xb] = v.reshape(zb - za, yb - ya, xb - xa)
        return g

    def corners(self, g):
        nx, ny, nz = (b[2] - 1 for b in self.box)
        return [g[q >> 2:(q >> 2) + nz, (q >> 1 & 1):(q >> 1 & 1) + ny, (q & 1):(q & 1) + nx] for q in range(8)]

    def rows(self, v):
        u = self.corners(self.grid(v))
        return [sum(self.kd[p ^ q] * u[q] for q in range(8)) for p in range(8)]

    def apply(self, v):
        (xa, xb, nx), (ya, yb, ny), (za, zb, nz) = self.box
        g = torch.zeros(nz, ny, nx, dtype=torch.float64, device="cuda")
        for part, r in zip(self.corners(g), self.rows(v)):
            part += self.k * r
        return g[za:zb, ya:yb, xa:xb].reshape(-1)

    def energy(self, lam, x):
        return sum(u * r for u, r in zip(self.corners(self.grid(lam)), self.rows(x)))


def _pcg(A, M, f):
    x = torch.zeros_like(f)
    r, p, rz = f.clone(), None, None
    for _ in range(1500):
        z = M(r)
        n = torch.dot(r, z)
        p = z if p is None else z + (n / rz) * p
        rz = n
        q = A(p)
        a = rz / torch.dot(p, q)
        x += a * p
        r -= a * q
        if float(r.norm()) < 1e-15 * float(f.norm()):
            break
    return x


def exact(case, seed):
    c = case
    kind = c["kind"]
    mats = _axis_matrices(c)
    shape = tuple(b - a for _, a, b in reversed(_axes(c)))
    if kind == "solve" or kind == "ensemble":
        members, W = c.get("members", 1), _warm(c)
        inv = _inverse(mats)
        out = []
        for j in range(members):
            f = _loads(c, seed, j, W + 1)[W]
            if not c["faces"]:
                f = f - f.mean()
            x = inv(f.reshape(shape)).reshape(-1)
            out.append((x if c["faces"] else x - x.mean()).cpu())
        return out[0] if kind == "solve" else torch.stack(out)
    if kind == "gradient":
        E = _Elements(c)
        inv = _inverse(mats)
        pre = lambda v: inv(v.reshape(shape)).reshape(-1)  # noqa: E731
        f = _loads(c, seed, 0, _warm(c) + 1)[_warm(c)]
        x = _pcg(E.apply, pre, f)
        lam = _pcg(E.apply, pre, x - _target(c, seed, 1e-2))
        return {"x": x.cpu(), "grad_f": lam.cpu(), "grad_g": (-E.k * E.energy(lam, x)).cpu()}
    KM, cut = _tensors(mats), torch.tensor(_cut(c), device="cuda")
    imats, (ix, iy, iz) = _interior(c, mats)
    inner = _inverse(imats)

    def interior(v):
        """K_II^{-1} of the interior values of v, zero on the interface."""
        w = torch.zeros_like(v)
        w[iz[:, None, None], iy[None, :, None], ix[None, None, :]] = inner(v[iz][:, iy][:, :, ix])
        return w

    def on_interface(x):
        v = torch.zeros(shape, dtype=torch.float64, device="cuda")
        v[cut] = x
        return v

    if kind in ("schur", "schur_batch"):
        X = _interface_input(c, seed, c.get("members", 1))
        Y = []
        for x in X:
            v = on_interface(x)
            Y.append(_apply(KM, v - interior(_apply(KM, v)))[cut].cpu())
        return Y[0] if kind == "schur" else torch.stack(Y)
    f = _loads(c, seed, 0, 1)[0].reshape(shape)
    v = on_interface(_interface_input(c, seed, 1)[0])
    b = f - _apply(KM, interior(f))
    return [b[cut].cpu(), (v + interior(f - _apply(KM, v))).reshape(-1).cpu()]
