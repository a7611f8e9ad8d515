"""dd_schur_apply_noalloc with the dense local solver (coefficient varying inside the subdomains): more
subdomains than SMs, and fewer, where the context's own product with K_II^{-1} is divided among several
CTAs per matrix. The entry point promises no shared state but its scratch array, so it also runs beside
dd_schur_apply of the same context on another stream. Tolerances of test_gpu_parity.py: FP64 1e-12 of
the largest entry, df64 1e-11.
"""
import ctypes

import numpy as np
import pytest

from workload import Mesh, graded_coords

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2412_17543_gb300 as P  # noqa: E402
from paper_2412_17543_gb300 import _native as nat  # noqa: E402


def _noalloc(S, x, y, stream):
    return S.lib.dd_schur_apply_noalloc(S.handle, ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(y.data_ptr()),
                                        ctypes.c_void_p(stream.cuda_stream))


@pytest.mark.parametrize("n,sub", [(24, 8), (24, 4)])  # 27 and 216 subdomains
@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("df64", 1e-11)])
def test_noalloc_dense(n, sub, prec, tol):
    c = graded_coords(n, 1.08, 20.0)[0]
    coef = np.exp(np.random.default_rng(5).standard_normal((n, n, n)))
    m = Mesh(n, n, n, c, c, c, (sub, sub, sub), 2, coef, "dense", {})
    S = P.Solver(m, levels=2, schur_prec=prec)
    assert S.info["local_solver"] == 1
    X = torch.as_tensor(np.random.default_rng(n).standard_normal((2, S.n_gamma)), device="cuda:0")
    ref = [S.schur_apply(X[j]) for j in range(2)]
    side, main = torch.cuda.Stream(), torch.cuda.current_stream()
    y = torch.full_like(X[0], float("nan"))
    assert _noalloc(S, X[0], y, main) == nat.DD_OK, S.lib.dd_last_error()
    torch.cuda.synchronize()
    assert (y - ref[0]).abs().max() <= tol * ref[0].abs().max()
    # sixteen calls queued on the side stream while the context applies its operator on the main one
    out = torch.full((16, S.n_gamma), float("nan"), dtype=torch.float64, device="cuda:0")
    torch.cuda.synchronize()
    for j in range(16):
        assert _noalloc(S, X[0], out[j], side) == nat.DD_OK
        assert torch.equal(S.schur_apply(X[1]), ref[1])
    torch.cuda.synchronize()
    for j in range(16):
        assert torch.equal(out[j], y)
    S.close()
