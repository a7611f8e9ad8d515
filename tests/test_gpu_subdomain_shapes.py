"""Subdomain operators on subdomain shapes at the edges of their ranges: one to eight elements per
axis, not cubes, Dirichlet data on several or no faces, varying coefficients (the dense local
solver's boundary block), ensembles whose members do not fill a chunk, and coarse spaces on both
sides of the size up to which the coarse operator is an explicit matrix.

Tolerances as in test_gpu_parity.py: FP64 operators 1e-12 of the largest entry (condensation and
recovery, which solve with K_II, 1e-11), df64 1e-11, FP32 BDDC 1e-4.
"""
import numpy as np
import pytest

from oracle import dd
from workload import Mesh, graded_coords, load_sequence, make_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2412_17543_gb300 as P  # noqa: E402

KINDS = (dd.CORNER, dd.EDGE, dd.FACE)
X0, X1, Y0, Z1 = 1, 2, 4, 32

# (elements per subdomain, subdomains per axis, Dirichlet faces)
SHAPES = {
    "6x4x5": ((6, 4, 5), (2, 3, 2), X0 | X1),
    "8x3x7": ((8, 3, 7), (2, 2, 2), X1 | Y0 | Z1),
    "1x8x2": ((1, 8, 2), (4, 2, 3), X1),       # subdomains without interior unknowns among them
    "8x8x8_one_axis": ((8, 8, 8), (3, 1, 1), X1),  # interior boxes of nine nodes
    "8x8x8_mid": ((8, 8, 8), (3, 3, 3), X1),
}
_cache = {}


def T(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


def N(t):
    torch.cuda.synchronize()
    return t.detach().cpu().numpy()


def case(name, coef=False):
    if (name, coef) not in _cache:
        s, b, faces = SHAPES[name]
        n = [s[a] * b[a] for a in range(3)]
        c = [graded_coords(v, 1.2, 20.0)[0] if v >= 4 else np.linspace(0.0, 1.0, v + 1) for v in n]
        k = None
        if coef:
            k = np.exp(np.random.default_rng(3).standard_normal((n[2], n[1], n[0])))
        m = Mesh(n[0], n[1], n[2], c[0], c[1], c[2], s, faces, k, name, {})
        _cache[name, coef] = (m, dd.q1_substructures(m))
    return _cache[name, coef]


def _solver(m, **kw):
    return P.Solver(m, levels=2, use_corners=1, use_edges=1, use_faces=1, weights="diag", **kw)


def _close(y, yo, tol):
    assert np.isfinite(y).all()
    assert np.abs(y - yo).max() <= tol * np.abs(yo).max()


@pytest.mark.parametrize("name", list(SHAPES))
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("df64", 1e-11)])
@pytest.mark.parametrize("coef", [False, True])
def test_single_operators(name, prec, tol, coef):
    m, subs = case(name, coef)
    S = _solver(m, schur_prec=prec)
    assert S.info["local_solver"] == (1 if coef else 2)
    rng = np.random.default_rng(1)
    x, f = rng.standard_normal(len(subs.gamma)), rng.standard_normal(S.n_free)
    _close(N(S.schur_apply(T(x))), subs.schur_apply(x), tol)
    _close(N(S.condense(T(f))), subs.condense(f), 1e-11)
    _close(N(S.recover(T(f), T(x))), subs.recover(f, x), 1e-11)
    S.close()


@pytest.mark.parametrize("name", ["6x4x5", "1x8x2", "8x8x8_one_axis", "8x8x8_mid"])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("df64", 1e-11)])
def test_ensemble_operators(name, prec, tol):
    """Calls of 9, 1 and 32 members on one context: members past the call's own count are padding."""
    m, subs = case(name)
    S = _solver(m, schur_prec=prec)
    for nrhs in (9, 1, 32):
        X = np.random.default_rng(nrhs).standard_normal((nrhs, len(subs.gamma)))
        Y = N(S.schur_apply_batch(T(X)))
        for j in range(nrhs):
            _close(Y[j], subs.schur_apply(X[j]), tol)
    S.close()


def test_ensemble_solves_of_changing_width():
    """A state used with 32, then 5, then 32 members: solutions as from single solves."""
    m, subs = case("8x8x8_mid")
    S = _solver(m, schur_prec="df64", precond_prec="fp32", flexible=1)
    rec = S.ensemble_recycler(4)
    for step, nrhs in enumerate((32, 5, 32)):
        F = np.stack([load_sequence(m, 60 + j, step + 1)[step] for j in range(nrhs)])
        X, st = S.solve_batch(T(F), rec, rtol=1e-10)
        X = N(X)
        for j in (0, nrhs // 2, nrhs - 1):
            x, _ = S.solve(T(F[j]), S.recycler(0), rtol=1e-10)
            x = N(x)
            assert np.linalg.norm(X[j] - x) <= 1e-8 * np.linalg.norm(x)
            assert st[j]["rel_res"] < 1e-10
    S.close()


@pytest.mark.parametrize("n,group,dense", [(16, 4, True), (20, 5, False)])
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("fp32", 1e-4)])
def test_coarse_operator_forms(n, group, dense, prec, tol):
    """2^3 subdomains: 2863 coarse dofs (explicit matrix) and 5859 (level by level), single and
    ensemble, against the oracle's three-level BDDC."""
    m = make_mesh(n, 2, 1.08, 20.0)
    subs = dd.q1_substructures(m)
    S = P.Solver(m, levels=3, coarse_group=group, use_corners=1, use_edges=1, use_faces=1, weights="diag",
                 precond_prec=prec)
    assert (S.info["n_coarse"] <= 4096) == dense
    Po = dd.Preconditioner(subs, 3, KINDS, "diag", group=group)
    R = np.random.default_rng(2).standard_normal((3, len(subs.gamma)))
    Z = N(S.precond_apply_batch(T(R)))
    for j in range(3):
        zo = Po.apply(R[j])
        _close(N(S.precond_apply(T(R[j]))), zo, tol)
        _close(Z[j], zo, tol)
    S.close()
