"""FGMRES queues the next Arnoldi step before it knows whether the present one ends the
cycle.  A queued step that is not needed costs a whole preconditioner, operator and
orthogonalisation: on grids where that is more than the host's wait, solves that their
tolerance ends after 1 to 20 steps launch no more kernels than with profiling on, which
queues nothing ahead; and on every grid they take the same steps."""
import numpy as np
import pytest

import scenes
from tests.gpu_common import need_gpu, problem_for, small_scene, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("dim,n", [(2, 33), (2, 300), (3, 24), (3, 44)])
def test_no_surplus_step(dim, n, precision):
    import paper_2405_12380_gb300 as hm
    s = small_scene(dim, n)
    P = problem_for(s, precision=precision)
    P.don_load(scenes.glorot_mlp(np.random.default_rng(5), [dim, 48, 48, 24]), 24, tau=1e-3)
    f = to_dev(s["b"])
    free = P.solve(f, None, hm.opts("fgmres", "rbgs", 2, tol=1e-14, restart=30, maxit=20))[1]["hist"]
    for steps in (1, 2, 3, 8, 20):
        o = hm.opts("fgmres", "rbgs", 2, tol=float(free[steps]) * (1 + 1e-3), restart=30, maxit=60)
        x, st = P.solve(f, None, o)
        P.set_profiling(True)
        xp, sp = P.solve(f, None, o)
        P.set_profiling(False)
        assert st["iters"] == sp["iters"], steps
        if n ** dim > 1 << 16:
            assert st["launches"] == sp["launches"], steps
        assert np.array_equal(x.cpu().numpy(), xp.cpu().numpy())
