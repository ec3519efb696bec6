"""The set union's sort (prefix-code keys, 2048-pair tiles, merge passes)
against numpy's lexicographic unique at the edges of its tiles and runs, on
rows that share long prefixes and on every byte value, for the three entry
points."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_13576_gb300 import mape
    mape.lib(build_if_missing=True)
    return mape


def _rows(kind, K, n, ldc, seed):
    rng = np.random.default_rng(seed)
    if kind == "bytes":      # every value, the code's length classes and -128 among them
        a = rng.integers(-128, 128, size=(K, n))
    elif kind == "sparse":   # mostly zeros: keys of about 30 coordinates, many of them equal
        a = rng.integers(-1, 2, size=(K, n)) * (rng.random((K, n)) < 0.05)
    elif kind == "prefix":   # equal up to the last few entries
        a = np.broadcast_to(rng.integers(-9, 10, size=n), (K, n)).copy()
        a[:, -3:] = rng.integers(-40, 41, size=(K, 3))
    else:                    # magnitudes around the code's class boundaries
        a = rng.choice([0, 1, 2, 3, 4, 7, 8, 15, 16, 31, 32, 63, 64, 127], size=(K, n)) * rng.choice([-1, 1], size=(K, n))
    out = np.zeros((K, ldc), np.int8)
    out[:, :n] = a
    return out


def _want(rows):
    u = np.unique(rows.astype(np.int16), axis=0)  # lexicographic on signed values
    return u.astype(np.int8)


@pytest.mark.parametrize("kind", ["bytes", "sparse", "prefix", "edges"])
@pytest.mark.parametrize("K", [1, 2, 7, 9, 255, 2047, 2048, 2049, 4097, 20000])
def test_sorted_union(M, kind, K):
    import torch
    for n, ldc in ((5, 16), (77, 80), (300, 304)):
        rows = _rows(kind, K, n, ldc, K + n)
        want = _want(rows)
        cand = torch.from_numpy(rows).cuda()
        got = M.dedup(cand, K, n).cpu().numpy()
        assert np.array_equal(got, want)
        uniq = torch.empty((K, ldc), dtype=torch.int8, device="cuda")
        k = ctypes.c_int64(0)
        rc = M.lib().mape_dedup_static(ctypes.c_void_p(cand.data_ptr()), K, n, ldc, ctypes.c_void_p(uniq.data_ptr()),
                                       K, ctypes.byref(k), None)
        assert rc == 0 and np.array_equal(uniq[: k.value].cpu().numpy(), want)


def test_uneven_sets_in_one_batch(M):
    import torch
    sizes = [(1, 5, 16), (2049, 77, 80), (0, 20, 32), (9000, 300, 304), (2048, 16, 16)]
    rows = [_rows("sparse" if i % 2 else "edges", K, n, ldc, 7 + i) for i, (K, n, ldc) in enumerate(sizes)]
    got = M.dedup_batch([(torch.from_numpy(np.concatenate([r, np.zeros((1, r.shape[1]), np.int8)])).cuda(), K, n, None)
                         for r, (K, n, _) in zip(rows, sizes)])
    for (g, k, status), r in zip(got, rows):
        assert status == 0 and k == _want(r).shape[0]
        assert np.array_equal(g.cpu().numpy(), _want(r))
