"""Profiling classes: the product with K_II^{-1} of the dense local solver is timed, and the byte counts of the
single sequence's iterations hold what the timed launches read and write.
"""
import numpy as np
import pytest

from workload import Mesh, graded_coords, load_sequence, make_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2412_17543_gb300 as P  # noqa: E402


def T(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda:0")


@pytest.mark.parametrize("prec", ["fp64", "df64"])
def test_kii_product_of_the_dense_solver_is_timed(prec):
    n = 16
    c = graded_coords(n, 1.08, 20.0)[0]
    coef = np.exp(np.random.default_rng(2).standard_normal((n, n, n)))
    S = P.Solver(Mesh(n, n, n, c, c, c, (8, 8, 8), 2, coef, "dense", {}), levels=2, schur_prec=prec)
    x = torch.ones(S.n_gamma, dtype=torch.float64, device="cuda:0")
    S.profile(True)
    for _ in range(3):
        S.schur_apply(x)
    prof, _ = S.profile(False)
    ms, launches, nbytes, _ = prof["KIIinv_apply"]
    assert launches == 3 and ms > 0.0 and nbytes > 0.0
    assert prof["schur_apply"][1] == 3 and prof["schur_apply"][0] >= ms
    S.close()


@pytest.mark.parametrize("flexible,k", [(0, 0), (1, 4)])
def test_bytes_of_the_iterations(flexible, k):
    """Against applications outside a solve, an iteration's Schur class also reads p and writes the histories of
    p and q, its BDDC class reads r (and z_old, flexible) and writes the history of z."""
    m = make_mesh(16, 4, 1.08, 20.0)
    S = P.Solver(m, levels=2, use_corners=1, use_edges=1, use_faces=1, flexible=flexible)
    v, n = torch.ones(S.n_gamma, dtype=torch.float64, device="cuda:0"), 8.0 * S.n_gamma
    S.profile(True)
    S.schur_apply(v)
    S.precond_apply(v)
    alone, _ = S.profile(True)
    rec = S.recycler(k)
    _, st = S.solve(T(load_sequence(m, 3, 1)[0]), rec, rtol=1e-8)
    its = st["iters"]
    prof, _ = S.profile(False)
    # without a basis: one application for the initial residual, then one per iteration; the iterations all
    # fit the histories of a recycler with k > 0. The recycling update, recorded in its own class, applies the
    # operators too
    assert 0 < its < 60
    assert prof["precond_apply"][1] >= its and prof["schur_apply"][1] >= its + 1
    kept = 1 if k else 0
    extra = (prof["schur_apply"][2] - alone["schur_apply"][2]) * prof["schur_apply"][1]
    assert extra == pytest.approx(its * n * (1 + 2 * kept), rel=1e-9)
    extra = (prof["precond_apply"][2] - alone["precond_apply"][2]) * prof["precond_apply"][1]
    assert extra == pytest.approx(its * n * (1 + flexible + kept), rel=1e-9)
    S.close()


def test_bytes_of_the_deflation():
    """k columns of A W (df64) and of W (FP64 preconditioner: df64), z and p in, p out; the Krylov dots are formed
    with z."""
    m = make_mesh(16, 4, 1.08, 20.0)
    S = P.Solver(m, levels=2, use_corners=1, use_edges=1, use_faces=1)
    rec = S.recycler(4)
    F = load_sequence(m, 3, 3)
    for t in range(2):
        S.solve(T(F[t]), rec, rtol=1e-8)
    S.profile(True)
    _, st = S.solve(T(F[2]), rec, rtol=1e-8)
    prof, _ = S.profile(False)
    assert st["recycled_k"] == 4 and prof["deflation"][1] == st["iters"]
    assert prof["deflation"][2] == pytest.approx((4 * 16.0 + 24.0) * S.n_gamma, rel=1e-12)
    S.close()
