"""The one-launch streamed extraction where its warps are kept apart: the first
step's debug outputs are written lane by lane between the tensor-memory loads,
with two blocks on every SM and more tiles than run at once.  The gradient
and the state are those of the step-by-step kernels, every time."""
import numpy as np
import pytest

from paper_2412_13576_gb300 import instances as I

from .test_gpu_cluster import M, _instance, _run  # noqa: F401  (M is the module fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,tiles,prec", [(1290, 258, 78, "PREC_FP8"), (1290, 258, 120, "PREC_BF16X1"),
                                            (1290, 258, 130, "PREC_BF16"), (487, 97, 150, "PREC_BF16")])
def test_debug_outputs_between_the_loads(M, n, m, tiles, prec):  # noqa: F811
    inst = _instance(n, m, 0.02)
    Z0 = I.normal_starts(inst, 128 * tiles - 3, std=0.3, seed=tiles).Z0
    want = _run(M, inst, Z0, getattr(M, prec), T=1, stepwise=True)
    for _ in range(4):
        got = _run(M, inst, Z0, getattr(M, prec), T=1)
        for k in ("grad", "Z", "M", "V", "rows"):
            assert np.array_equal(got[k], want[k]), k
