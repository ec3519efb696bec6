"""The projection of samples to coordinates at the edges of its kernels: the
64-wide blocks of the factorisation, the ring of staged rows (16-byte copies
for d % 4 == 0, single words otherwise, a shorter ring for d > 3632) and the
128 x 64 output tiles, against a 64-bit Cholesky solve.  Bound per start: that
of the FP32 factorisation and solves, 8 d cond(B^T B) 2^-24; for B = [I; -C]
the condition number is at most 1 + |C|_2^2."""
import numpy as np
import pytest

from paper_2412_13576_gb300 import instances as I

from .gpu_common import dev, per_start_rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_13576_gb300 import mape
    mape.lib(build_if_missing=True)
    return mape


@pytest.mark.parametrize("d,m,P,density", [
    (1, 1, 1, None), (2, 3, 5, None), (31, 7, 127, 0.3), (63, 9, 128, 0.2), (64, 8, 129, 0.2), (65, 1, 33, 0.2),
    (127, 30, 64, 0.1), (128, 20, 200, 0.1), (129, 44, 257, 0.1), (514, 37, 130, 0.02), (3632, 21, 3, 0.004),
    (3700, 40, 130, 0.004),
])
def test_project_edges(M, d, m, P, density):
    from scipy.linalg import cho_factor, cho_solve
    inst = I.make_instance("edges", d + m, m, c_k=1, c_density=density, lo=-3, hi=3, q_k=1, q_density=0.0, lin_k=1,
                           seed=d)
    G0 = I.uniform_samples(inst, P, seed=5).G0
    Z = M.project_starts(dev(inst.B), dev(G0)).cpu().numpy()
    B = inst.B.astype(np.float64)
    Zo = cho_solve(cho_factor(B.T @ B), B.T @ G0.T.astype(np.float64)).T
    bound = 8 * d * (1 + np.linalg.norm(B[d:], 2) ** 2) * 2.0 ** -24
    err = per_start_rel(Z, Zo)
    assert err.max() < bound, (err.max(), bound)
