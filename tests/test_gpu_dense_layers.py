"""Element-wise and reduction kernels of the dense layers at the sizes where their
vector width, their cluster split and their tails change, and on arrays that are not
16-byte aligned, against FP64 numpy.  A sum of n FP32 products in any order differs
from the exact one by at most n 2^-24 of the sum of magnitudes."""
import ctypes as C

import numpy as np
import pytest

from tests.gpu_common import need_gpu, to_dev, torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


def _lib():
    from paper_2405_12380_gb300 import _lib as L
    return L.lib()


def _p(t):
    # (data_ptr() of an empty tensor is null, which the calls refuse)
    return C.c_void_p(t.untyped_storage().data_ptr() + 4 * t.storage_offset())


def _off(a, off):
    """A device copy of `a` that starts `off` floats past an aligned address."""
    t = torch.empty(a.size + off + 1, dtype=torch.float32, device="cuda")
    t[off:off + a.size] = to_dev(a.reshape(-1))
    return t[off:off + a.size]


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("rows,cols", [(1, 1), (7, 3), (255, 33), (256, 32), (257, 100), (300, 31), (5000, 260), (0, 5)])
def test_bias_grad(rows, cols, off):
    dY = np.random.default_rng(rows + cols).standard_normal((rows, cols)).astype(np.float32)
    d, db = _off(dY, off), torch.full((cols,), 7.0, device="cuda")
    assert _lib().nn_bias_grad(rows, cols, _p(d), _p(db), None) == 0
    err = np.abs(db.cpu().numpy() - dY.astype(np.float64).sum(0))
    assert np.all(err <= max(rows, 1) * U * np.abs(dY).astype(np.float64).sum(0))


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("B,P2", [(1, 1), (3, 4095), (2, 4096), (5, 4097), (4, 4099), (33, 20000)])
def test_rel_l2(B, P2, off):
    rng = np.random.default_rng(B + P2)
    pr, tg = (rng.standard_normal((B, P2)).astype(np.float32) for _ in range(2))
    a, b = _off(pr, off), _off(tg, off)
    d, lo = torch.empty(B * P2, device="cuda"), torch.empty(B, device="cuda")
    assert _lib().nn_rel_l2(B, P2, _p(a), _p(b), _p(d), _p(lo), None) == 0
    df, t64 = pr.astype(np.float64) - tg, tg.astype(np.float64)
    den = (t64 ** 2).sum(1)
    loss = (df ** 2).sum(1) / den
    assert np.all(np.abs(lo.cpu().numpy() - loss) <= (2 * P2 + 8) * U * loss)
    ref = 2.0 / (den[:, None] * B) * df
    err = np.abs(d.cpu().numpy().reshape(B, P2) - ref)
    scale = 2.0 / (den[:, None] * B) * (np.abs(pr) + np.abs(tg))      # the subtraction rounds once
    assert np.all(err <= (P2 + 8) * U * np.abs(ref) + 2 * U * scale)


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("n", [0, 1, 3, 4, 1027, 70001])
def test_adam_and_act_backward(n, off):
    rng = np.random.default_rng(n)
    p, g, m = (rng.standard_normal(n).astype(np.float32) for _ in range(3))
    v = rng.uniform(0, 2, n).astype(np.float32)
    P, G, M, V = (_off(a, off) for a in (p, g, m, v))
    lr, t = 1e-3, 7
    assert _lib().nn_adam(n, _p(P), _p(G), _p(M), _p(V), lr, 0.9, 0.999, 1e-8, t, None) == 0
    m1 = 0.9 * m.astype(np.float64) + 0.1 * g
    v1 = 0.999 * v.astype(np.float64) + 0.001 * g.astype(np.float64) ** 2
    # 1 - beta and 1 - beta^t carry the FP32 rounding of beta: up to 2^-24 / 1e-3 relative
    assert np.all(np.abs(M.cpu().numpy() - m1) <= 4 * U * (np.abs(m) + np.abs(g)))
    assert np.all(np.abs(V.cpu().numpy() - v1) <= 4 * U * v + 1e-4 * 0.001 * g ** 2)
    step = lr * (m1 / (1 - 0.9 ** t)) / (np.sqrt(v1 / (1 - 0.999 ** t)) + 1e-8)
    assert np.all(np.abs(P.cpu().numpy() - (p - step)) <= 2 * U * np.abs(p) + 1e-3 * np.abs(step) + 8 * U * lr * 10)
    for act in (0, 1, 2, 3):
        d, y = _off(g, off), _off(np.tanh(m), off)
        assert _lib().nn_act_backward(n, _p(d), _p(y), act, None) == 0
        y64 = np.tanh(m).astype(np.float64)
        f = [np.ones_like(y64), y64 > 0, 1 - y64 * y64, np.where(y64 > 0, 1.0, 0.01)][act]
        assert np.all(np.abs(d.cpu().numpy() - g * f) <= 4 * U * np.abs(g))


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("rows,cols", [(1, 1), (3, 4), (5, 255), (4099, 256), (2, 1028), (33, 70000)])
def test_bias_act(rows, cols, off):
    rng = np.random.default_rng(rows * 3 + cols)
    X, b = rng.standard_normal((rows, cols)).astype(np.float32), rng.standard_normal(cols).astype(np.float32)
    for act, f in ((0, lambda z: z), (1, lambda z: np.maximum(z, 0)), (2, np.tanh), (3, lambda z: np.where(z > 0, z, 0.01 * z))):
        x, bb = _off(X, off), _off(b, 1 - off)
        assert _lib().nn_bias_act(rows, cols, _p(x), _p(bb), act, None) == 0
        ref = f(X.astype(np.float64) + b)
        assert np.all(np.abs(x.cpu().numpy().reshape(rows, cols) - ref) <= 4 * U * (np.abs(X) + np.abs(b) + 1e-6))
    x = _off(X, off)
    assert _lib().nn_bias_act(rows, cols, _p(x), None, 1, None) == 0
    assert np.array_equal(x.cpu().numpy().reshape(rows, cols), np.maximum(X, 0))


@pytest.mark.parametrize("ta", [0, 1])
@pytest.mark.parametrize("tb", [0, 1])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (33, 129, 15), (64, 128, 16), (65, 257, 17), (32, 256, 4101), (128, 128, 300),
                                   (130, 3, 2049), (5, 700, 128)])
def test_gemm_tiles(ta, tb, M, N, K):
    """Edges of the GEMM's tiles (32 and 128 rows, 128 and 256 columns), slabs and K
    splits, leading dimensions with and without 16-byte rows, beta 0, 1 and general.
    |C - exact| <= (K + 4) 2^-24 (|A| |B|) + a few ulps of beta C."""
    rng = np.random.default_rng(M + 3 * N + 7 * K)
    for pad, beta in ((0, 0.0), (4 - (M + N + K) % 4, 1.0), (1, -0.75)):
        A = rng.standard_normal((K, M + pad) if ta else (M, K + pad)).astype(np.float32)
        B = rng.standard_normal((N, K + pad) if tb else (K, N + pad)).astype(np.float32)
        C0 = rng.standard_normal((M, N + pad)).astype(np.float32)
        opA = (A[:, :M].T if ta else A[:, :K]).astype(np.float64)
        opB = (B[:, :K].T if tb else B[:, :N]).astype(np.float64)
        Ad, Bd, Cd = _off(A, pad % 2), to_dev(B), to_dev(C0)
        if beta == 0.0:
            Cd[:, :N] = float("nan")                      # not read
        assert _lib().nn_gemm(ta, tb, M, N, K, 1.5, _p(Ad), A.shape[1], _p(Bd), B.shape[1], beta, _p(Cd), N + pad, None) == 0
        got = Cd.cpu().numpy()
        ref = 1.5 * (opA @ opB) + beta * C0[:, :N]
        bound = (K + 4) * U * 1.5 * (np.abs(opA) @ np.abs(opB)) + 4 * U * abs(beta) * np.abs(C0[:, :N])
        assert np.all(np.abs(got[:, :N] - ref) <= bound)
        assert np.array_equal(got[:, N:], C0[:, N:])      # nothing outside the matrix


@pytest.mark.parametrize("ta,tb", [(0, 0), (0, 1), (1, 0), (1, 1)])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (16, 128, 64), (17, 129, 65), (33, 300, 128), (65, 128, 1000), (129, 20000, 64),
                                   (3, 5, 5000)])
def test_gemm_bf16_tiles(ta, tb, M, N, K):
    """Edges of the BF16 product's tiles (16 to 128 rows of C by 128 columns), of the
    conversion's 64 x 64 blocks and of the ring (fewer K steps than stages, and wrapping
    it), leading dimensions with and without 16-byte rows, beta 0 with NaN in C and general:
    |C - exact| <= 4 K 2^-24 (|A| |B|) on the rounded operands, as in test_gpu_gemm_tc.py."""
    from oracle.tb import bf16_round
    rng = np.random.default_rng(M + 3 * N + 7 * K)
    for pad, beta in ((0, 0.0), (1, -0.75)):
        A = rng.standard_normal((K, M + pad) if ta else (M, K + pad)).astype(np.float32)
        B = rng.standard_normal((N, K + pad) if tb else (K, N + pad)).astype(np.float32)
        C0 = rng.standard_normal((M, N + pad)).astype(np.float32)
        opA = bf16_round((A[:, :M].T if ta else A[:, :K]).astype(np.float64))
        opB = bf16_round((B[:, :K].T if tb else B[:, :N]).astype(np.float64))
        Ad, Bd, Cd = _off(A, pad), to_dev(B), to_dev(C0)
        if beta == 0.0:
            Cd[:, :N] = float("nan")
        assert _lib().nn_gemm_bf16(ta, tb, M, N, K, 1.5, _p(Ad), A.shape[1], _p(Bd), B.shape[1], beta, _p(Cd), N + pad, None) == 0
        got = Cd.cpu().numpy()
        bound = 4 * K * U * 1.5 * (np.abs(opA) @ np.abs(opB)) + 4 * U * abs(beta) * np.abs(C0[:, :N]) + 1e-30
        assert np.all(np.abs(got[:, :N] - (1.5 * (opA @ opB) + beta * C0[:, :N])) <= bound)
        assert np.array_equal(got[:, N:], C0[:, N:])
    flag = C.c_int(-1)
    assert _lib().nn_gemm_bf16_status(C.byref(flag)) == 0 and flag.value == 0


@pytest.mark.parametrize("N", [256, 4096, 8192, 16384])   # tiles of 16, 32, 64 and 128 rows
@pytest.mark.parametrize("K", [100, 192, 450, 833])        # 2, 3, 8 and 14 K steps: stages filled, part filled, reused
def test_gemm_bf16_stages(N, K):
    """Stages of several K steps, the last one part filled: bound as in test_gemm_bf16_tiles."""
    from oracle.tb import bf16_round
    M = 128
    rng = np.random.default_rng(N + K)
    A, B = rng.standard_normal((M, K)).astype(np.float32), rng.standard_normal((N, K)).astype(np.float32)
    opA, opB = bf16_round(A.astype(np.float64)), bf16_round(B.T.astype(np.float64))
    Ad, Bd, Cd = to_dev(A), to_dev(B), to_dev(np.full((M, N), np.nan, np.float32))
    assert _lib().nn_gemm_bf16(0, 1, M, N, K, 1.0, _p(Ad), K, _p(Bd), K, 0.0, _p(Cd), N, None) == 0
    assert np.all(np.abs(Cd.cpu().numpy() - opA @ opB) <= 4 * K * U * (np.abs(opA) @ np.abs(opB)) + 1e-30)
    flag = C.c_int(-1)
    assert _lib().nn_gemm_bf16_status(C.byref(flag)) == 0 and flag.value == 0


@pytest.mark.parametrize("rows,cols", [(0, 5), (1, 1), (31, 8), (33, 9), (1024, 100), (1025, 33), (5000, 20)])
def test_bias_grad_rows_keeps_the_order(rows, cols):
    """The sums in the order of the rows, bit for bit (one tile of 1024 rows, its edges, several)."""
    dY = np.random.default_rng(rows + cols).standard_normal((max(rows, 1), cols)).astype(np.float32)
    ref = np.zeros(cols, np.float32)
    for r in range(rows):
        ref += dY[r]
    Dd, db = to_dev(dY), to_dev(np.full(cols, np.nan, np.float32))
    assert _lib().nn_bias_grad_rows(rows, cols, _p(Dd), _p(db), None) == 0
    assert np.array_equal(db.cpu().numpy(), ref)


def test_adam_same_bits_on_every_path():
    """Values in 16-byte groups, in the tail and in arrays off 16 bytes take the same step."""
    rng = np.random.default_rng(9)
    a = [rng.standard_normal(4099).astype(np.float32) for _ in range(3)] + [rng.random(4099).astype(np.float32)]
    out = []
    for off in (0, 1):
        for n in (4099, 4096):
            d = [_off(x[-n:], off) for x in a]
            assert _lib().nn_adam(n, _p(d[0]), _p(d[1]), _p(d[2]), _p(d[3]), 1e-3, 0.9, 0.999, 1e-8, 4, None) == 0
            out.append([t.cpu().numpy()[-4096:] for t in d])
    for o in out[1:]:
        for x, y in zip(out[0], o):
            assert np.array_equal(x, y)
