"""The kernel test and the coefficients over tiles of 32 transposed rows, and
the routes beside them (rows of A with a large absolute sum; directions at any
pitch), against numpy in 64 bits at the edges of the tile, of its 16-byte
pieces, of the entry chunks and of the packed 16-bit sums.  Integers: equal."""
import numpy as np
import pytest

from .gpu_common import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_13576_gb300 import mape
    mape.lib(build_if_missing=True)
    return mape


def _pitched(M, G, n):
    buf = np.full((G.shape[0], M.round16(n)), -77, np.int8)  # the pitch's tail holds anything
    buf[:, :n] = G
    return buf


@pytest.mark.parametrize("m,n,K", [(1, 257, 1), (33, 300, 31), (200, 260, 33), (5, 1000, 100), (70, 2500, 64),
                                   (9, 4096, 65), (20, 1280, 40), (12, 1536, 33)])
@pytest.mark.parametrize("big", [False, True])
def test_kernel_test_tiles(M, m, n, K, big):
    rng = np.random.default_rng(m + n + K + big)
    d = n - m
    C = rng.integers(-2, 3, size=(m, d)) * (rng.random((m, d)) < min(1.0, 20.0 / d))
    z = rng.integers(-1, 2, size=(K, d)) * (rng.random((K, d)) < 0.5)
    A = np.concatenate([C, np.eye(m, dtype=np.int64)], axis=1)
    G = np.concatenate([z, -(z @ C.T)], axis=1)
    assert np.abs(G).max() <= 127
    # single entries off, and rows at the ends of int8
    for k in range(0, K, 3):
        G[k, rng.integers(n)] += rng.choice([-1, 1])
    if K > 8:
        G[4], G[5] = -128, 127
        G[6], G[7] = np.where(A[0] > 0, -128, 127), np.where(A[0] > 0, 127, -128)
    # one row of A at the largest sum of the packed route, or past it: 512 x (-128) = -2^16
    A[0] = 0
    A[0, :128] = 4 if big else 2
    A[0, 0] -= 0 if big else 1
    assert np.abs(A[0]).sum() == (512 if big else 255)
    want = np.all(G.astype(np.int64) @ A.T == 0, axis=1)
    ok, fails = M.kernel_test(dev(A.astype(np.int32)), dev(_pitched(M, G, n)), n)
    assert np.array_equal(ok.cpu().numpy().astype(bool), want) and fails == int((~want).sum())


@pytest.mark.parametrize("m,n", [(3100, 17), (3100, 16), (1600, 31), (800, 64)])
def test_kernel_test_full_rows(M, m, n):
    """Rows of A without zeros, where a fill to a multiple of four has no room."""
    rng = np.random.default_rng(m + n)
    A = np.tile(rng.choice([-2, -1, 1, 2], size=(1, n)), (m, 1))
    A[m // 2:] *= -1
    G = rng.integers(-3, 4, size=(70, n))
    for k in range(0, 70, 2):      # an exact row: the last entries take up the sum
        G[k, -2:] = 0
        r = int(G[k] @ A[0])
        G[k, -1] = -r // A[0, -1] if r % A[0, -1] == 0 else 0
    want = np.all(G @ A.T == 0, axis=1)
    assert want.any() and not want.all()
    ok, fails = M.kernel_test(dev(A.astype(np.int32)), dev(_pitched(M, G, n)), n)
    assert np.array_equal(ok.cpu().numpy().astype(bool), want) and fails == int((~want).sum())


@pytest.mark.parametrize("n,K,nnz", [(1, 1, 1), (15, 31, 0), (16, 32, 100), (17, 33, 1023), (100, 64, 1024),
                                     (1000, 70, 1025), (1024, 33, 500), (4096, 40, 5000)])
@pytest.mark.parametrize("quartic,small", [(False, False), (True, False), (True, True)])
@pytest.mark.parametrize("pitched", [True, False])
def test_coeffs_tiles(M, n, K, nnz, quartic, small, pitched):
    rng = np.random.default_rng(n + K + nnz)
    G = rng.integers(-3, 4, size=(K, n))
    G[:, 0] = -128
    G[K // 2] = rng.choice([-128, 127], size=n)
    G[0] = -128
    qr = rng.integers(0, n, size=nnz).astype(np.int32)
    qc = np.maximum(qr, rng.integers(0, n, size=nnz)).astype(np.int32)
    # values at the ends of a chunk's 32-bit sums, and past them
    qv = (rng.choice([-4095, 4095], size=nnz) if small else rng.integers(-2 ** 31, 2 ** 31, size=nnz)).astype(np.int32)
    w = rng.integers(0, 2 ** 20, size=n).astype(np.int32) if quartic else None
    g = G.astype(np.int64)
    f = np.where(qr == qc, 1, 2) * qv.astype(np.int64)
    want_a = (g[:, qr] * g[:, qc]) @ f if nnz else np.zeros(K, np.int64)
    want_q = (g ** 4) @ w.astype(np.int64) if quartic else np.zeros(K, np.int64)
    rows = _pitched(M, G, n) if pitched else G.astype(np.int8)
    a, q4 = M.direction_coeffs(dev(qr), dev(qc), dev(qv), None if w is None else dev(w), n, dev(rows))
    assert np.array_equal(a.cpu().numpy(), want_a) and np.array_equal(q4.cpu().numpy(), want_q)
