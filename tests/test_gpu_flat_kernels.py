"""FP64 kernels that take nodes in the flat order (operator, residual and norm, Jacobi and
red-black sweeps, the red-row residual) on grids whose rows and planes do not divide into
warps and blocks, 3 to 66 nodes a side, conj, with and without a stored k^2 field, against
the oracle (tolerances of test_gpu_parity.py); and the integer conversion between FP64 and
FP32 pairs over exponents on both sides of its range: the trunk-basis correction is linear
and powers of two are exact, so a scaled right-hand side gives the scaled correction up to
the pairs' 2^-48 (times the correction's condition, below 1e3 here)."""
import numpy as np
import pytest

import scenes
from oracle import assemble, relax
from tests.gpu_common import need_gpu, problem_for, rel, small_scene, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("field", [False, True])
@pytest.mark.parametrize("dim,n", [(2, 3), (2, 31), (2, 66), (3, 3), (3, 4), (3, 16), (3, 17), (3, 33), (3, 50), (3, 66)])
def test_operator_and_sweeps(dim, n, field):
    s = small_scene(dim, n, cells=1 if n < 9 else 4, box=(1, 0) if n < 5 else None)
    A0, k2 = s["A"], None
    if field:
        k2 = assemble.k2_field(dim, n, s["k0"], s["cells"], 0.5, 1.0 + 0.05 * s["rng"].standard_normal(n ** dim))
        A0 = assemble.assemble(dim, n, k2, s["mask"])
    P = problem_for(s, k2=k2)
    x = s["rng"].standard_normal(n ** dim) + 1j * s["rng"].standard_normal(n ** dim)
    col = assemble.colour(dim, n)
    for conj in (0, 1):
        A = A0.conj() if conj else A0
        assert rel(P.apply(to_dev(x), conj=conj).cpu().numpy(), A @ x) < 1e-13
        r, nrm = P.residual(to_dev(s["b"]), to_dev(x), conj=conj)
        ref = s["b"] - A @ x
        assert rel(r.cpu().numpy(), ref) < 1e-13
        assert abs(nrm.item() - np.vdot(ref, ref).real) <= 1e-12 * np.vdot(ref, ref).real
        for kind, fn in (("rbgs", lambda: relax.rbgs(A, s["b"], x, col, 2)), ("sor", lambda: relax.sor(A, s["b"], x, col, 1.3, 2)),
                         ("jacobi", lambda: relax.jacobi(A, s["b"], x, 1.3, 2))):
            y = P.relax(kind, to_dev(s["b"]), to_dev(x), sweeps=2, omega=1.3, conj=conj)
            assert rel(y.cpu().numpy(), fn()) < 1e-12, kind


@pytest.mark.parametrize("e", [-70, -40, 60, 100])
def test_pair_conversion_over_exponents(e):
    n = 21
    s = small_scene(3, n)
    P = problem_for(s)
    P.don_load(scenes.glorot_mlp(np.random.default_rng(3), [3, 32, 32, 16]), 16, tau=1e-3)
    r = s["rng"].standard_normal(n ** 3) + 1j * s["rng"].standard_normal(n ** 3)
    r *= 10.0 ** s["rng"].uniform(-3, 0, n ** 3)
    r[s["mask"] == 1] = 0
    z = P.don_correct(to_dev(r)).cpu().numpy()
    zs = P.don_correct(to_dev(np.ldexp(r.real, e) + 1j * np.ldexp(r.imag, e))).cpu().numpy()
    assert rel(np.ldexp(zs.real, -e) + 1j * np.ldexp(zs.imag, -e), z) < 1e3 * 2.0 ** -44
    bad = r.copy()
    bad[5 * n * n + 5 * n + 5] = np.inf
    assert not np.isfinite(P.don_correct(to_dev(bad)).cpu().numpy()).all()
