"""Dense layers with as many rows or columns as their int arguments hold: the strides of the
row and column loops must not run past 2^31.  (Blocks of 8.6 GB, one element wide.)"""
import pytest

from tests.gpu_common import need_gpu, torch

pytestmark = pytest.mark.gpu
BIG = 2 ** 31 - 1


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()
    if torch.cuda.get_device_properties(0).total_memory < 64e9:
        pytest.skip("needs 64 GB of device memory")
    yield
    torch.cuda.empty_cache()


def _call(fn, *args):
    from paper_2405_12380_gb300 import _lib
    p = [a.data_ptr() if torch.is_tensor(a) else a for a in args]
    assert getattr(_lib.lib(), fn)(*p, torch.cuda.current_stream().cuda_stream) == 0
    torch.cuda.synchronize()


@pytest.mark.parametrize("rows,cols", [(BIG, 1), (1, BIG), (1, BIG - 3), (BIG - 4000, 1)])
def test_bias_act(rows, cols):
    X = torch.full((rows * cols,), -1.0, device="cuda")
    bias = torch.full((cols,), 3.0, device="cuda")
    _call("nn_bias_act", rows, cols, X, bias, 1)
    assert bool((X == 2).all())


@pytest.mark.parametrize("rows,cols", [(BIG, 1), (3, BIG // 3), (1, BIG)])
def test_bias_grad(rows, cols):
    d = torch.ones(rows * cols, device="cuda")
    db = torch.full((cols,), -1.0, device="cuda")
    _call("nn_bias_grad", rows, cols, d, db)
    assert float((db - rows).abs().max()) <= 1e-6 * rows


@pytest.mark.parametrize("P2", [BIG, BIG - 255])
def test_rel_l2(P2):
    pred, target = torch.full((P2,), 2.0, device="cuda"), torch.ones(P2, device="cuda")
    loss = torch.zeros(1, device="cuda")
    d = torch.zeros(P2, device="cuda")
    _call("nn_rel_l2", 1, P2, pred, target, d, loss)
    assert abs(float(loss) - 1) < 1e-5
    assert float((d * P2 - 2).abs().max()) < 1e-4
