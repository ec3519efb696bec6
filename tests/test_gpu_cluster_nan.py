"""The one-launch streamed extraction from a start whose first coordinate is NaN
(the maximum of |z| is NaN then) and whose others lie beyond 2^22, where
adding and subtracting 1.5 2^23 does not round: the bits of the step-by-step
kernels, as for every start."""
import numpy as np
import pytest

from paper_2412_13576_gb300 import instances as I

from .test_gpu_cluster import M, _instance, _same  # noqa: F401  (M is the module fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["PREC_BF16", "PREC_BF16X1", "PREC_FP8"])
def test_nan_first_and_large_coordinates(M, prec):  # noqa: F811
    inst = _instance(100, 20, 0.2)
    Z0 = I.normal_starts(inst, 40, std=0.4, seed=4).Z0.astype(np.float32)
    big = np.float32([8388609.0, -8388611.0, 16777215.0, 4194305.0, -4194305.5])
    for r in range(0, 32, 3):  # of the starts of a warp some, not all
        Z0[r, 0] = np.nan
        Z0[r, 5:10] = big
        Z0[r, -5:] = -big
    _same(M, inst, Z0, getattr(M, prec), T=3)
