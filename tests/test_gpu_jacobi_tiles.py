"""Several 2D Jacobi sweeps per launch: sweep counts around the launch size (one launch,
several, odd and even from a given x), grids of one ragged tile, of ragged last tiles, at
the largest size of the tiled form and just above it; complex128 and complex64, conj, and
a stored k^2 field, against the oracle's sweeps.  The sweeps contract (omega = 0.6), so
each adds a few units in the last place: 1e-12 in FP64 as in test_gpu_parity.py, and 20
2^-24 a sweep in complex64."""
import numpy as np
import pytest

from oracle import assemble, relax
from tests.gpu_common import need_gpu, problem_for, rel, small_scene, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("field", [False, True])
@pytest.mark.parametrize("n", [5, 13, 64, 73, 193, 384, 385])
def test_tiled_sweeps_match_oracle(n, field):
    s = small_scene(2, n, cells=1 if n < 9 else 4)
    k2 = None
    A0 = s["A"]
    if field:
        k2 = assemble.k2_field(2, n, s["k0"], s["cells"], 0.5, 1.0 + 0.05 * s["rng"].standard_normal(n * n))
        A0 = assemble.assemble(2, n, k2, s["mask"])
    P = problem_for(s, k2=k2)
    x0 = s["rng"].standard_normal(n * n) + 1j * s["rng"].standard_normal(n * n)
    for conj in (0, 1):
        A, ref, done = (A0.conj() if conj else A0), x0, 0
        for sweeps in (1, 2, 4, 5, 6, 11, 20):
            ref = relax.jacobi(A, s["b"], ref, 0.6, sweeps - done)
            done = sweeps
            x = P.relax("jacobi", to_dev(s["b"]), to_dev(x0), sweeps=sweeps, omega=0.6, conj=conj)
            assert rel(x.cpu().numpy(), ref) < 1e-12, sweeps
            x = P.relax("jacobi", to_dev(s["b"], torch.complex64), to_dev(x0, torch.complex64), sweeps=sweeps, omega=0.6,
                        conj=conj)
            assert rel(x.cpu().numpy(), ref) < 20 * sweeps * 2.0 ** -24 + 2.0 ** -22, sweeps
