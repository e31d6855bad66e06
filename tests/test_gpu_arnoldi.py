"""The Arnoldi step's kernels at the sizes where their tiles and groups change: fewer
nodes than a 32-row tile, a ragged last tile, 64- to 256-row tiles, one to 64 basis
vectors (several row groups per vector, one vector per lane, more vectors than a warp),
in FP64 (same iterate as the oracle, the tolerance of test_gpu_parity.py: CGS2 in FP64
keeps FGMRES's iterates to rounding) and on mixed handles (the product widened inside).
The step queued ahead of the one that ends a solve must leave the solution alone."""
import numpy as np
import pytest

from oracle import krylov
from tests.gpu_common import need_gpu, problem_for, rel, small_scene, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("dim,n,restart,maxit", [(2, 5, 3, 3), (2, 9, 1, 4), (2, 9, 15, 15), (2, 33, 16, 17), (2, 65, 33, 40),
                                                 (3, 13, 64, 64), (3, 21, 31, 32), (3, 45, 8, 20)])
def test_fgmres_same_iterate_over_tiles(dim, n, restart, maxit):
    import paper_2405_12380_gb300 as hm
    s = small_scene(dim, n, cells=1 if n < 9 else 4)
    P = problem_for(s)
    o = hm.opts("fgmres", "none", 0, correction="none", tol=1e-300, restart=restart, maxit=maxit)
    x, st = P.solve(to_dev(s["b"]), None, o)
    x0 = np.where(s["mask"] == 1, s["b"], 0)
    xo, io = krylov.fgmres(s["A"], s["b"], x0, None, 1e-300, restart, maxit)
    if io["est"][-1] > 1e-12:                       # (not solved exactly within the steps)
        assert st["iters"] == io["iters"] and st["precond_applies"] == io["iters"]
        assert np.allclose(st["hist"][1:], io["est"], rtol=1e-7, atol=0)
    assert rel(x.cpu().numpy(), xo) < 1e-10


@pytest.mark.parametrize("precision,tol", [("fp64", 1e-6), ("mixed", 1e-3)])
def test_stop_inside_a_cycle(precision, tol):
    """Ended by its tolerance in the middle of a cycle (the next step is already queued),
    the solution is that of the step that met it: the true residual equals the estimate."""
    import paper_2405_12380_gb300 as hm
    s = small_scene(3, 20)
    P = problem_for(s, precision=precision)
    x, st = P.solve(to_dev(s["b"]), None, hm.opts("fgmres", "rbgs", 2, correction="none", tol=tol, restart=60, maxit=400))
    assert st["status"] == 0 and st["iters"] % 60 != 0
    b = s["b"]
    res = np.linalg.norm(b - s["A"] @ x.cpu().numpy()) / np.linalg.norm(b)
    assert res <= tol and abs(res - st["rel_res"]) <= 1e-6 * res
    if precision == "fp64" and st["iters"] < 60:
        assert abs(res - st["hist"][st["iters"]]) <= 1e-6 * res
    # the same steps as a budget instead of a tolerance
    y, st2 = P.solve(to_dev(b), None, hm.opts("fgmres", "rbgs", 2, correction="none", tol=1e-300, restart=60,
                                              maxit=st["iters"]))
    assert st2["iters"] == st["iters"] and rel(y.cpu().numpy(), x.cpu().numpy()) < 1e-12
