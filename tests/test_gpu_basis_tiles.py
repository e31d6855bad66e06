"""The trunk-basis setup where the Gram matrix's 16 x 16 tiles and the columns of the
basis product change shape (one column, a full and a ragged tile, several tiles, more
columns than a tile row of threads), against the oracle, with the tolerances of
test_gpu_parity.py's setup test: at tau = 1e-3 the kept columns' condition (about 1e3 to
1e5) times the FP64 rounding of the Gram matrix stays below 1e-9."""
import numpy as np
import pytest

import scenes
from oracle import tb as otb
from tests.gpu_common import need_gpu, problem_for, rel, small_scene

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("n,width,p", [(13, 32, 1), (21, 32, 15), (21, 32, 16), (21, 32, 17), (13, 64, 33), (21, 130, 130)])
def test_setup_matches_oracle(n, width, p):
    s = small_scene(3, n)
    layers = scenes.glorot_mlp(np.random.default_rng(p), [3, width, width, p])
    P = problem_for(s)
    k = P.don_load(layers, p, tau=1e-3)
    so = otb.tb_setup(s["A"], layers, scenes.node_coords(3, n), s["mask"], p, tau=1e-3)
    assert P.kept == so.kept
    Q = P.basis().cpu().numpy()
    assert np.max(np.abs(Q.T @ Q - np.eye(k))) < 1e-13
    assert rel(Q, so.Q) < 1e-9
    assert rel(P.coarse_inverse().cpu().numpy(), np.linalg.inv(so.Ac)) < 1e-9
