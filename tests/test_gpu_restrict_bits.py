"""The order of the FP32 sums in the complex64 restriction and the roundings of the residual
it projects, bit for bit against a numpy restatement of the whole cycle: red rows on odd and
2D grids (one partial tile, several blocks, more partial rows than threads) and all rows
after Jacobi, SOR and no sweeps, column counts that are not a multiple of a warp's, the
absorbing layer and a stored k^2, conj."""
import numpy as np
import pytest

import scenes
from oracle import assemble
from tests.f32_cycle import Op32, pair
from tests.gpu_common import need_gpu, problem_for, small_scene, to_dev, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("field", [False, True])
@pytest.mark.parametrize("dim,n,p", [(2, 20, 9), (2, 45, 17), (2, 300, 40), (3, 13, 8), (3, 20, 24), (3, 37, 33), (3, 105, 6)])
def test_order_of_the_sums(dim, n, p, field):
    import paper_2405_12380_gb300 as hm
    s = small_scene(dim, n)
    N = n ** dim
    k2 = assemble.k2_field(dim, n, s["k0"], s["cells"], 0.5, 1.0 + 0.05 * s["rng"].standard_normal(N)) if field else None
    op = Op32(dim, n, s["k0"], s["mask"], s["cells"], k2=k2)
    P = problem_for(s, precision="mixed", k2=k2)
    P.don_load(scenes.glorot_mlp(np.random.default_rng(5), [dim, 48, 48, p]), p, tau=1e-3)
    Q, Ainv = P.basis().cpu().numpy(), P.coarse_inverse().cpu().numpy()
    r = s["rng"].standard_normal(N) + 1j * s["rng"].standard_normal(N)
    r[s["mask"] == 1] = 0
    r = r.astype(np.complex64)
    rd = to_dev(r, torch.complex128)
    for kind, n_r in [("none", 0), ("jacobi", 2), ("rbgs", 1), ("sor", 1)]:
        if kind == "rbgs" and dim == 3 and n % 2 == 0:
            continue                                       # the pair layout has an order of its own
        for conj in (False, True):
            cyc = lambda c: pair(P.precond(rd, hm.opts("fgmres", kind, n_r, omega=0.8, correction=c, conj=conj)).cpu().numpy())  # noqa: E731
            want = op.cycle(Q, Ainv, pair(r), cyc("none") if n_r else None, kind == "rbgs", conj)
            assert all(np.array_equal(a, b) for a, b in zip(cyc("tb"), want)), (kind, conj)
