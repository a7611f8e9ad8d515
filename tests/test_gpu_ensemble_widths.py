"""A recycle state of an ensemble used with changing member counts: every count's PCG loop is captured once, and
the solutions are those of single solves."""
import numpy as np
import pytest

from workload import load_sequence, make_mesh

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

import paper_2412_17543_gb300 as P  # noqa: E402

WIDTHS = (12, 32, 1, 20)


@pytest.mark.parametrize("local,prec", [("fdm", "df64"), ("fdm", "fp64"), ("dense", "fp64")])
def test_changing_widths_are_captured_once(local, prec):
    m = make_mesh(16, 8 if local == "fdm" else 4, 1.08, 20.0)
    S = P.Solver(m, levels=2, use_corners=1, use_edges=1, use_faces=1, schur_prec=prec, local_solver=local)
    F = torch.as_tensor(np.stack([load_sequence(m, 70 + j, 1)[0] for j in range(32)]), device="cuda:0")
    rec = S.ensemble_recycler(0)
    one = S.recycler(0)
    want = [S.solve(F[j].contiguous(), one, rtol=1e-11)[0] for j in range(32)]

    def run():
        for w in WIDTHS:
            X, _ = S.solve_batch(F[:w].contiguous(), rec, rtol=1e-11)
            for j in {0, w // 2, w - 1}:
                assert (X[j] - want[j]).norm() <= 1e-8 * want[j].norm()

    def calls():
        with torch.profiler.profile(activities=[torch.profiler.ProfilerActivity.CPU,
                                                torch.profiler.ProfilerActivity.CUDA]) as prof:
            run()
            torch.cuda.synchronize()
        return [e.key for e in prof.key_averages()]

    calls()  # captures; a process's first profile does not hold every call
    names = calls()
    assert any("cudaGraphLaunch" in n for n in names)
    assert not any("Instantiate" in n or "BeginCapture" in n for n in names)
    S.close()


@pytest.mark.parametrize("fdm_rc", [4, 8])
def test_members_per_block(fdm_rc):
    """Counts that do and do not fill a block against single applications (df64: 1e-11 of the largest entry), and the
    reported shapes: what the kernel runs with."""
    m = make_mesh(16, 8, 1.3, 20.0)
    S = P.Solver(m, levels=2, use_corners=1, use_edges=1, use_faces=1, schur_prec="df64", local_solver="fdm",
                 ens_fdm_rc=fdm_rc)
    X = torch.as_tensor(np.random.default_rng(fdm_rc).standard_normal((32, S.n_gamma)), device="cuda:0")
    Y = torch.stack([S.schur_apply(x) for x in X])
    for w in (1, 3, 4, 5, 8, 9, 31, 32):
        Z = S.schur_apply_batch(X[:w].contiguous())
        assert ((Z - Y[:w]).abs().amax(dim=1) <= 1e-11 * Y[:w].abs().amax(dim=1)).all()
    assert (S.info["ens_elem_rc"], S.info["ens_fdm_rc"]) == (fdm_rc, fdm_rc)
    S.close()
