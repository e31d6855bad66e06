"""The roundings of complex64 damped-Jacobi sweeps, bit for bit: 2D grids that take several
sweeps per launch (one ragged tile, ragged last tiles, the largest of them) and the first
that takes one, and 3D; from zero and from a given x, sweep counts around the launch size,
the absorbing layer and a stored k^2, conj.  How many sweeps share a launch must not show."""
import numpy as np
import pytest

from oracle import assemble
from tests.f32_cycle import Op32, pair
from tests.gpu_common import need_gpu, problem_for, small_scene, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("field", [False, True])
@pytest.mark.parametrize("dim,n", [(2, 13), (2, 64), (2, 193), (2, 768), (2, 769), (3, 20), (3, 21)])
def test_roundings_of_the_sweeps(dim, n, field):
    import paper_2405_12380_gb300 as hm
    s = small_scene(dim, n)
    N = n ** dim
    k2 = assemble.k2_field(dim, n, s["k0"], s["cells"], 0.5, 1.0 + 0.05 * s["rng"].standard_normal(N)) if field else None
    op = Op32(dim, n, s["k0"], s["mask"], s["cells"], k2=k2)
    P = problem_for(s, precision="mixed", k2=k2)
    f, x = (s["rng"].standard_normal(N) + 1j * s["rng"].standard_normal(N) for _ in range(2))
    f, x = f.astype(np.complex64), (x / n ** 2).astype(np.complex64)
    for conj in (False, True):
        for sweeps in (1, 2, 5, 6, 11) if n < 700 else (6,):
            o = hm.opts("fgmres", "jacobi", sweeps, omega=0.6, correction="none", conj=conj)
            z = pair(P.precond(to_dev(f, torch.complex128), o).cpu().numpy())
            want = op.jacobi(0.6, sweeps, pair(f), None, conj)
            assert all(np.array_equal(a, b) for a, b in zip(z, want)), ("from zero", conj, sweeps)
            y = pair(P.relax("jacobi", to_dev(f), to_dev(x), sweeps=sweeps, omega=0.6, conj=conj).cpu().numpy())
            want = op.jacobi(0.6, sweeps, pair(f), pair(x), conj)
            assert all(np.array_equal(a, b) for a, b in zip(y, want)), ("from x", conj, sweeps)
