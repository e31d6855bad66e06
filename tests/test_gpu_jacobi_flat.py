"""Damped-Jacobi sweeps of complex128 at a launch a sweep: 2D grids above the tiled form and
3D grids, with ragged last blocks and an odd number of planes, the absorbing layer and a
stored k^2, from x and from zero, conj: the oracle's sweeps, to the tolerance of
test_gpu_jacobi_tiles.py."""
import numpy as np
import pytest

from oracle import assemble, relax
from tests.gpu_common import need_gpu, problem_for, rel, small_scene, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("dim,n", [(2, 161), (2, 992), (2, 999), (2, 1000), (2, 1021), (2, 1025), (3, 100), (3, 126), (3, 127)])
def test_sweeps_match_oracle(dim, n):
    import paper_2405_12380_gb300 as hm
    s = small_scene(dim, n)
    N = n ** dim
    k2 = assemble.k2_field(dim, n, s["k0"], s["cells"], 0.5, 1.0 + 0.05 * s["rng"].standard_normal(N)) if n % 2 else None
    A = s["A"] if k2 is None else assemble.assemble(dim, n, k2, s["mask"])
    P = problem_for(s, k2=k2)
    x0 = s["rng"].standard_normal(N) + 1j * s["rng"].standard_normal(N)
    x = P.relax("jacobi", to_dev(s["b"]), to_dev(x0), sweeps=3, omega=0.6).cpu().numpy()
    assert rel(x, relax.jacobi(A, s["b"], x0, 0.6, 3)) < 1e-12
    z = P.precond(to_dev(s["b"]), hm.opts("fgmres", "jacobi", 2, omega=0.6, correction="none", conj=True)).cpu().numpy()
    assert rel(z, relax.jacobi(A.conj(), s["b"], np.zeros_like(x0), 0.6, 2)) < 1e-12
