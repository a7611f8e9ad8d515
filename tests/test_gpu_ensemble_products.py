"""Ensemble BDDC where its launch shapes and forms change: local matrices of 1 to 16 block rows (one warp per block row
up to eight, else sixteen), and coarse spaces small enough for the ensemble to apply the explicit coarse matrix (1115
dofs, not a multiple of the rows of a block or of the columns of a chunk). Against the oracle, tolerances of
test_gpu_ensemble.py: FP64 1e-10 of the largest entry, FP32 1e-4.
"""
import numpy as np
import pytest

from oracle import dd
from workload import Mesh, graded_coords, load_sequence

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2412_17543_gb300 as P  # noqa: E402

KINDS = (dd.CORNER, dd.EDGE, dd.FACE)
_cache = {}


def T(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


def N(t):
    torch.cuda.synchronize()
    return t.detach().cpu().numpy()


def case(n, s):
    if (n, s) not in _cache:
        c = [graded_coords(v, 1.08, 20.0)[0] for v in n]
        m = Mesh(n[0], n[1], n[2], c[0], c[1], c[2], (s, s, s), 2, None, "products", {})
        _cache[n, s] = (m, dd.q1_substructures(m))
    return _cache[n, s]


def _solver(m, levels, group, **kw):
    return P.Solver(m, levels=levels, coarse_group=group, use_corners=1, use_edges=1, use_faces=1, weights="diag", **kw)


def _close(y, yo, tol):
    assert np.isfinite(y).all()
    assert np.abs(y - yo).max() <= tol * np.abs(yo).max()


@pytest.mark.parametrize("n,s", [((12, 9, 12), 3), ((15, 10, 15), 5), ((18, 12, 12), 6), ((14, 14, 21), 7)])
@pytest.mark.parametrize("prec,nmm,tol", [("fp64", "auto", 1e-10), ("fp32", "simt", 1e-4)])
def test_local_products(n, s, prec, nmm, tol):
    m, subs = case(n, s)
    S = _solver(m, 2, 2, precond_prec=prec, ens_nmm=nmm)
    Po = dd.Preconditioner(subs, 2, KINDS, "diag")
    R = np.random.default_rng(s).standard_normal((5, len(subs.gamma)))
    Z = N(S.precond_apply_batch(T(R)))
    for j in range(5):
        _close(Z[j], Po.apply(R[j]), tol)
    S.close()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-10), ("fp32", 1e-4)])
@pytest.mark.parametrize("group", [2, 3])
def test_explicit_coarse_matrix(group, prec, tol):
    m, subs = case((12, 12, 12), 2)
    S = _solver(m, 3, group, precond_prec=prec)
    assert 1024 < S.info["n_coarse"] <= 2048 and S.info["n_coarse"] % 8
    Po = dd.Preconditioner(subs, 3, KINDS, "diag", group=group)
    R = np.random.default_rng(group).standard_normal((9, len(subs.gamma)))
    Z = N(S.precond_apply_batch(T(R)))
    for j in range(9):
        _close(Z[j], Po.apply(R[j]), tol)
    S.close()


def test_solve_with_the_explicit_coarse_matrix():
    m, _ = case((12, 12, 12), 2)
    S = _solver(m, 3, 3, schur_prec="df64", precond_prec="fp32", flexible=1)
    rec = S.ensemble_recycler(4)
    for step in range(3):
        F = np.stack([load_sequence(m, 80 + j, step + 1)[step] for j in range(11)])
        X, st = S.solve_batch(T(F), rec, rtol=1e-10)
        X = N(X)
        for j in (0, 5, 10):
            x = N(S.solve(T(F[j]), S.recycler(0), rtol=1e-10)[0])
            assert np.linalg.norm(X[j] - x) <= 1e-8 * np.linalg.norm(x)
            assert st[j]["rel_res"] < 1e-10
    S.close()
