"""FGMRES is homogeneous in its right-hand side and powers of two are exact, so the estimates
relative to it are the same for a right-hand side of any size, down to where the square of
its norm is still a normal number and far below that for the estimates themselves."""
import numpy as np
import pytest

from tests.gpu_common import need_gpu, problem_for, small_scene, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("e", [-490, -300, 300, 490])
def test_estimates_over_scales(e):
    import paper_2405_12380_gb300 as hm
    s = small_scene(2, 9)
    P = problem_for(s)
    o = hm.opts("fgmres", "none", 0, correction="none", tol=1e-300, restart=60, maxit=60)
    ref = P.solve(to_dev(s["b"]), None, o)[1]["hist"]
    got = P.solve(to_dev(np.ldexp(s["b"].real, e) + 1j * np.ldexp(s["b"].imag, e)), None, o)[1]["hist"]
    n = int(np.argmax(ref < 1e-14)) or len(ref)          # (the solve is exact after as many steps as nodes)
    assert n > 20 and ref[n - 1] < 1e-5
    assert np.allclose(got[:n], ref[:n], rtol=1e-9, atol=0)
