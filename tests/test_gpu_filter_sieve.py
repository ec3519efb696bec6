"""The minimality filter's choice of dense coordinates (6 for the lists, the
next 32 for the pair test) around the row lengths where there are not enough of
them, with ties among the counts and dense coordinates at either end, and its
scan four rows at a time, against the brute-force minimal set; alone and as
one batch.  Flags and rows: equal."""
import numpy as np
import pytest

from oracle import mape_oracle as O

from .gpu_common import dev
from .test_gpu_stages import _planted_dense

pytestmark = pytest.mark.gpu

SHAPES = [(40, 1), (300, 3), (500, 6), (500, 7), (600, 37), (601, 38), (602, 39), (603, 64), (700, 65), (500, 130),
          (7, 200)]


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_13576_gb300 import mape
    mape.lib(build_if_missing=True)
    return mape


def _rows(M, K, n):
    rng = np.random.default_rng(31 * K + n)
    if n == 1:
        G = np.arange(1, K + 1)[:, None]
    else:
        G = _planted_dense(rng, K, n)
    thin = rng.random(n) < 0.5          # half the coordinates sparse: the dense ones are spread over the row
    G = G * np.where(thin[None, :], rng.random(G.shape) < 0.2, True)
    G = G[np.any(G != 0, axis=1)]
    G = np.unique(np.array([O.canonical_sign(g) for g in G]), axis=0)
    buf = np.full((G.shape[0], M.round16(n)), 77, np.int8)  # the pitch's tail holds anything
    buf[:, :n] = G
    valid = (rng.random(G.shape[0]) < 0.9).astype(np.uint8)
    expect = np.zeros(G.shape[0], bool)
    expect[valid != 0] = O.minimal_elements(G[valid != 0])
    return buf, valid, expect


@pytest.mark.parametrize("K,n", SHAPES)
def test_dense_coordinates_and_scan(M, K, n):
    buf, valid, expect = _rows(M, K, n)
    keep, out = M.minimal_filter(dev(buf), n, valid=dev(valid))
    assert np.array_equal(keep.cpu().numpy().astype(bool), expect)
    assert np.array_equal(out.cpu().numpy()[:, :n], buf[expect][:, :n])


def test_dense_coordinates_batch(M):
    cases = [_rows(M, K, n) for K, n in SHAPES]
    got = M.minimal_filter_batch([(dev(b), n, dev(v)) for (b, v, _), (_, n) in zip(cases, SHAPES)])
    for (b, _, expect), (_, n), (keep, out) in zip(cases, SHAPES, got):
        assert np.array_equal(keep.cpu().numpy().astype(bool), expect)
        assert np.array_equal(out.cpu().numpy()[:, :n], b[expect][:, :n])
