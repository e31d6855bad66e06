"""FP32 products whose K is not split are one chain of fused multiply-adds a value, bit for
bit against numpy: short K at a few rows and at many, long K with C on either side of the
size from which it is not split, one tile an SM and more, both transpositions.  (A split K
is added atomically, in an order that changes from call to call.)"""
import numpy as np
import pytest

from tests.f32_cycle import chain
from tests.gpu_common import need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


@pytest.mark.parametrize("M,N,K", [(32, 100, 100), (32, 256, 127), (65, 33, 96), (256, 256, 100), (4864, 256, 130),
                                   (5000, 256, 256), (9900, 70, 127), (9728, 128, 140), (11000, 100, 140)])
def test_unsplit_product_is_one_chain(M, N, K):
    from paper_2405_12380_gb300 import _lib
    lib = _lib.lib()
    rng = np.random.default_rng(M + N + K)
    A, B = rng.standard_normal((M, K)).astype(np.float32), rng.standard_normal((N, K)).astype(np.float32)
    want = chain(A.T[:, :, None], B.T[:, None, :])
    for tA, tB in ((0, 1), (1, 0)):
        a, b = (torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (A.T if tA else A, B if tB else B.T))
        c = torch.full((M, N), float("nan"), device="cuda")
        assert lib.nn_gemm(tA, tB, M, N, K, 1.0, a.data_ptr(), a.shape[1], b.data_ptr(), b.shape[1], 0.0, c.data_ptr(), N,
                           torch.cuda.current_stream().cuda_stream) == 0
        assert np.array_equal(c.cpu().numpy(), want), (tA, tB)
