"""The kernel test over tiles of 32 transposed rows, and the route beside it
(rows of A with a large absolute sum), against numpy in 64 bits at the edges of
the tile, of its 16-byte pieces and of the packed 16-bit sums.  Integers: equal."""
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
                                   (9, 4096, 65)])
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
