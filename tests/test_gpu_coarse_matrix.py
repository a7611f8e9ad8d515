"""The explicit coarse operator of small coarse spaces in an FP32 preconditioner: an application to a single
vector may be no further from the FP64 one than the products that the matrix stands for (through them 0.8e-7 to
1.8e-7, 2-norm, mean of three vectors).

Tolerance: an application takes four FP32 operators (Phi^T, the coarse operator, Phi, N_i). Entries, input and
sums of each are rounded once, independently, u / sqrt(3) each (u = 2^-24), which is u per operator and
2 u for the four; half as much again for cancellation makes 3 u.
"""
import pytest

from workload import Mesh, graded_coords

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2412_17543_gb300 as P  # noqa: E402

U = 2.0 ** -24
# (elements, elements per subdomain, group): 2863 and 573 coarse dofs; 1321 dofs, 1115 of them inside one level-2
# subdomain, whose matrix is wider than the FP64 tiles that form the others
MESHES = {"16^3 of 2^3": ((16, 16, 16), (2, 2, 2), 4), "30x24x20 of 6x4x5": ((30, 24, 20), (6, 4, 5), 2),
          "14x12x12 of 2^3, groups of 6": ((14, 12, 12), (2, 2, 2), 6)}


def _mesh(n, sub):
    c = [graded_coords(v, 1.08, 20.0)[0] for v in n]
    return Mesh(n[0], n[1], n[2], c[0], c[1], c[2], sub, 2, None, "coarse", {})


def _solver(m, group, prec, **kw):
    return P.Solver(m, levels=3, coarse_group=group, use_corners=1, use_edges=1, use_faces=1, weights="diag",
                    precond_prec=prec, **kw)


def _vectors(S):
    """Three random interface vectors and three in the range of A on smooth ones."""
    g = torch.Generator(device="cuda:0").manual_seed(7)
    R = torch.randn(6, S.n_gamma, dtype=torch.float64, device="cuda:0", generator=g)
    for j in range(3, 6):
        t = torch.linspace(0.0, 1.0 + j, S.n_gamma, dtype=torch.float64, device="cuda:0")
        R[j] = S.schur_apply(torch.sin(t))
    return R


def _mean_error(Z, E):
    e = ((Z - E).norm(dim=1) / E.norm(dim=1)).cpu().numpy()
    return float(e[:3].mean()), float(e[3:].mean())


@pytest.mark.parametrize("name", list(MESHES))
def test_fp32_application_is_as_near_fp64_as_the_products(name):
    n, sub, group = MESHES[name]
    m = _mesh(n, sub)
    S64, S32 = _solver(m, group, "fp64"), _solver(m, group, "fp32")
    assert S32.info["n_coarse"] <= 4096
    R = _vectors(S64)
    E = torch.stack([S64.precond_apply(r) for r in R])
    for e in _mean_error(torch.stack([S32.precond_apply(r) for r in R]), E):
        assert e <= 3 * U
    S64.close()
    S32.close()
