"""df64 Schur applications on the assembled rows against the FP64 operator (which is an order nearer the exact
one): single vectors within one df64 unit, 2^-48 in the 2-norm, with either local solver; ensembles, whose rows
have two chains instead of three and whose line contractions add their chains unnormalized, within 1.25 units. The
brick-by-brick form of the same products stood at 0.65 to 0.75 units (single) and 1.15 to 1.3 (ensembles) on such
meshes.
"""
import pytest

from workload import Mesh, graded_coords

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2412_17543_gb300 as P  # noqa: E402

UNIT = 2.0 ** -48


@pytest.mark.parametrize("n,s", [((35, 28, 42), 7), ((20, 20, 20), 5)])
@pytest.mark.parametrize("local", ["fdm", "dense"])
def test_df64_rows(n, s, local):
    c = [graded_coords(v, 1.08, 20.0)[0] for v in n]
    m = Mesh(n[0], n[1], n[2], c[0], c[1], c[2], (s, s, s), 2, None, "rows", {})
    kw = dict(levels=2, use_corners=1, use_edges=1, use_faces=1, weights="diag")
    S, E = P.Solver(m, schur_prec="df64", local_solver=local, **kw), P.Solver(m, schur_prec="fp64", **kw)
    g = torch.Generator(device="cuda:0").manual_seed(s)
    X = torch.randn(8, S.n_gamma, dtype=torch.float64, device="cuda:0", generator=g)
    R = torch.stack([E.schur_apply(x) for x in X])
    one = torch.stack([S.schur_apply(x) for x in X])
    assert ((one - R).norm(dim=1) / R.norm(dim=1)).mean().item() <= UNIT
    if local == "fdm":  # a dense K_II^{-1} serves FP64 ensembles only
        assert ((S.schur_apply_batch(X) - R).norm(dim=1) / R.norm(dim=1)).mean().item() <= 1.25 * UNIT
    S.close()
    E.close()
