"""Complex64 Gauss-Seidel sweeps that store one colour between two sweeps: from a given x
(one sweep packs that colour first) and from zero, one to four sweeps (each buffer in turn,
the full result last), layered and stored k^2, on grids of one warp a row, of two with a
ragged last one and of three, against the oracle's FP64 sweeps (tolerance of
test_gpu_sweep.py: a few units of 2^-24 a sweep)."""
import numpy as np
import pytest

from oracle import assemble, relax
from tests.gpu_common import need_gpu, problem_for, rel, small_scene, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("field", [False, True])
@pytest.mark.parametrize("n", [6, 22, 64, 66, 98, 130])
def test_sweeps_match_oracle(n, field):
    import paper_2405_12380_gb300 as hm
    s = small_scene(3, n, cells=min(4, n // 3))
    k2, A = None, s["A"]
    if field:
        k2 = assemble.k2_field(3, n, s["k0"], s["cells"], 0.5, 1.0 + 0.05 * s["rng"].standard_normal(n ** 3))
        A = assemble.assemble(3, n, k2, s["mask"])
    col = assemble.colour(3, n)
    x0 = s["rng"].standard_normal(n ** 3) + 1j * s["rng"].standard_normal(n ** 3)
    P = problem_for(s, k2=k2)
    Pm = problem_for(s, precision="mixed") if not field else None
    for sweeps in (1, 2, 3, 4) if n < 100 else (3,):
        for conj in (False, True) if n < 70 else (False,):
            Ac = A.conj() if conj else A
            x = P.relax("rbgs", to_dev(s["b"], torch.complex64), to_dev(x0, torch.complex64), sweeps=sweeps, conj=conj)
            assert rel(x.cpu().numpy(), relax.rbgs(Ac, s["b"], x0, col, sweeps)) < 3e-6 * sweeps, (sweeps, conj)
        if Pm:
            z = Pm.precond(to_dev(s["b"]), hm.opts("bicgstab", "rbgs", sweeps, correction="none"))
            assert rel(z.cpu().numpy(), relax.rbgs(A, s["b"], np.zeros_like(x0), col, sweeps)) < 3e-6 * sweeps, sweeps
