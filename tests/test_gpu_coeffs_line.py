"""The coefficients on both sides of the line between rows per warp and tiles of
32 transposed rows (entries of Q and twice the coordinates), at the edges of
the tiles: exact integers against numpy."""
import numpy as np
import pytest

from .gpu_common import dev
from .test_gpu_rows_tile import M  # noqa: F401  (the module fixture)

pytestmark = pytest.mark.gpu

LINE = 1850


@pytest.mark.parametrize("n", [1, 15, 16, 17, 33, 257, 925])
@pytest.mark.parametrize("past", [-1, 0, 1400])
@pytest.mark.parametrize("K", [1, 32, 67])
@pytest.mark.parametrize("quartic", [False, True])
def test_both_sides(M, n, past, K, quartic):  # noqa: F811
    rng = np.random.default_rng(n + past + K)
    nnz = max(0, LINE - 2 * n + past)
    rows = rng.integers(-128, 128, size=(K, M.round16(n))).astype(np.int8)
    g = rows[:, :n].astype(np.int64)
    qr = rng.integers(0, n, size=nnz).astype(np.int32)
    qc = np.maximum(qr, rng.integers(0, n, size=nnz)).astype(np.int32)
    qv = rng.integers(-5000, 5001, size=nnz).astype(np.int32)
    w = rng.integers(0, 9, size=n).astype(np.int32) if quartic else None
    f = qv.astype(np.int64) * np.where(qr == qc, 1, 2)
    want = (g[:, qr] * g[:, qc]) @ f if nnz else np.zeros(K, np.int64)
    a, q4 = M.direction_coeffs(dev(qr), dev(qc), dev(qv), None if w is None else dev(w), n, dev(rows))
    assert np.array_equal(a.cpu().numpy(), want)
    assert np.array_equal(q4.cpu().numpy(), (g ** 4) @ w.astype(np.int64) if quartic else np.zeros(K, np.int64))
