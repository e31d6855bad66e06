"""The roundings of the fused complex64 red-black sweep, bit for bit, in every form of the
kernel: from zero and from a given x, Gauss-Seidel, SOR and SSOR, the absorbing layer and
a stored k^2, conj, one and three sweeps, on grids of one ragged warp a row and of two.  A
solution in mixed precision moves by up to a hundred times what the cycle's rounding moves
by, so a change of the last bits here shows up in the fifth digit of a solve."""
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
@pytest.mark.parametrize("kind", ["rbgs", "sor", "ssor"])
@pytest.mark.parametrize("n", [20, 66])
def test_roundings_of_the_sweep(n, kind, field):
    import paper_2405_12380_gb300 as hm
    s = small_scene(3, n)
    k2 = assemble.k2_field(3, n, s["k0"], s["cells"], 0.5, 1.0 + 0.05 * s["rng"].standard_normal(n ** 3)) if field else None
    op = Op32(3, n, s["k0"], s["mask"], s["cells"], k2=k2)
    P = problem_for(s, precision="mixed", k2=k2)
    f, x = (s["rng"].standard_normal(n ** 3) + 1j * s["rng"].standard_normal(n ** 3) for _ in range(2))
    f, x = f.astype(np.complex64), (x / n ** 2).astype(np.complex64)
    for conj in (False, True):
        for sweeps in (1, 3) if n < 50 else (2,):
            o = hm.opts("fgmres", kind, sweeps, omega=1.2, correction="none", conj=conj)
            z = pair(P.precond(to_dev(f, torch.complex128), o).cpu().numpy())
            want = op.sweeps(kind, 1.2, sweeps, pair(f), None, conj)
            assert all(np.array_equal(a, b) for a, b in zip(z, want)), ("from zero", conj, sweeps)
            y = pair(P.relax(kind, to_dev(f), to_dev(x), sweeps=sweeps, omega=1.2, conj=conj).cpu().numpy())
            want = op.sweeps(kind, 1.2, sweeps, pair(f), pair(x), conj)
            assert all(np.array_equal(a, b) for a, b in zip(y, want)), ("from x", conj, sweeps)
