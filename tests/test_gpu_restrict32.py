"""The complex64 cycle's restriction after every kind of sweep (the red rows after
red-black Gauss-Seidel, all rows otherwise, the plain vector without sweeps) on odd and
even grids in 2D and 3D -- the residual is stored and then projected, 1024 rows a warp, so
grids of one ragged range, and of more ranges than a block holds, are among them --
against the oracle's cycle with the rounded basis (tolerance of test_gpu_mixed.py)."""
import numpy as np
import pytest

import scenes
from oracle import assemble, relax, tb as otb
from tests.gpu_common import need_gpu, problem_for, rel, small_scene, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("kind", ["none", "jacobi", "rbgs", "sor"])
@pytest.mark.parametrize("dim,n,p", [(2, 20, 9), (2, 45, 17), (3, 13, 8), (3, 20, 16), (3, 37, 24)])
def test_cycle_matches_oracle(dim, n, p, kind):
    import paper_2405_12380_gb300 as hm
    s = small_scene(dim, n)
    layers = scenes.glorot_mlp(np.random.default_rng(5), [dim, 48, 48, p])
    P = problem_for(s, precision="mixed")
    k = P.don_load(layers, p, tau=1e-3)
    so = otb.tb_setup(s["A"], layers, scenes.node_coords(dim, n), s["mask"], p, tau=1e-3)
    sm = otb.mixed_setup(so, s["A"])
    assert k == len(sm.kept)
    r = s["rng"].standard_normal(n ** dim) + 1j * s["rng"].standard_normal(n ** dim)
    r[s["mask"] == 1] = 0
    n_r = 0 if kind == "none" else 2
    z = P.precond(to_dev(r), hm.opts("fgmres", kind, n_r, omega=0.8)).cpu().numpy()
    col = assemble.colour(dim, n)
    z0 = {"none": np.zeros_like(r), "jacobi": relax.jacobi(s["A"], r, np.zeros_like(r), 0.8, n_r),
          "rbgs": relax.rbgs(s["A"], r, np.zeros_like(r), col, n_r),
          "sor": relax.sor(s["A"], r, np.zeros_like(r), col, 0.8, n_r)}[kind]
    assert rel(z, z0 + otb.tb_correct(sm, r - s["A"] @ z0)) < 1e-4
