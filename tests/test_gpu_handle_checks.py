"""The exact checks of a handle, A B = 0 at creation and A x = b before
Algorithm 1, at the edges of their blocks (128 columns of B, 1024 entries of a
row listed at once, eight rows of A to a block): one entry off is refused
wherever it lies, the right data is accepted."""
import dataclasses

import numpy as np
import pytest

from paper_2412_13576_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_13576_gb300 import mape
    mape.lib(build_if_missing=True)
    return mape


@pytest.mark.parametrize("n,m,density", [(2, 1, None), (33, 8, 0.5), (137, 9, None), (1024, 17, 0.05),
                                         (1025, 7, None), (2100, 3, 0.9)])
def test_one_entry_off(M, n, m, density):
    inst = I.make_instance("checks", n, m, c_k=1, c_density=density, lo=-4, hi=5, q_k=1, q_density=0.001, lin_k=1,
                           seed=n)
    cfg = M.default_config(T=2)
    d = n - m
    for i, j in ((0, 0), (n - 1, d - 1), (d, d // 2)):
        B = inst.B.copy()
        B[i, j] += 1
        if np.all(inst.A.astype(np.int64) @ B == 0):  # the column still lies in the kernel
            continue
        with pytest.raises(M.MapeError) as e:
            M.Instance.from_generated(dataclasses.replace(inst, B=B), cfg)
        assert e.value.code == -3
    with M.Instance.from_generated(inst, cfg) as h:
        h.extract_directions(8, Z0=I.normal_starts(inst, 8, std=0.3, seed=1).Z0)
        h.wait(60)
        X = np.repeat(inst.xbar[None, :], 3, axis=0)
        for r in {0, m // 2, m - 1}:
            bad = X.copy()
            bad[2, d + r] += 1 if bad[2, d + r] < inst.u[d + r] else -1  # A = [C | I]: row r alone is off
            with pytest.raises(M.MapeError) as e:
                h.augment(bad)
            assert e.value.code == -5
        h.augment(X)
        h.wait(60)
        assert np.array_equal(inst.A.astype(np.int64) @ h.solution()[0], inst.b)
