"""The one-launch streamed extraction at the lines of the rule that chooses the
blocks per tile and at the numbers of tiles beyond what runs at once (15 and 16,
36 and 37, 74 to 77, 152 and 153 tiles; a second and a third wave), where
tiles wait for an SM, and over enough steps for the state ring to turn some
hundred times: the bits of the step-by-step kernels."""
import pytest

from paper_2412_13576_gb300 import instances as I

from .test_gpu_cluster import M, _instance, _run  # noqa: F401  (M is the module fixture)

pytestmark = pytest.mark.gpu

import numpy as np  # noqa: E402


def _same(M, inst, Z0, prec, one_launch=True, **kw):  # noqa: F811
    a = _run(M, inst, Z0, prec, **kw)
    b = _run(M, inst, Z0, prec, stepwise=True, **kw)
    assert (a["launches"] < b["launches"]) == one_launch
    for k in ("Z", "M", "V", "grad", "rows"):
        assert a[k].shape == b[k].shape, k
        at = np.argwhere(a[k] != b[k])
        assert len(at) == 0, (k, len(at), at[:3].tolist(), at[-3:].tolist())
    assert a["flags"] == b["flags"]


@pytest.mark.parametrize("n,tiles", [(40, 15), (40, 16), (40, 36), (40, 37), (60, 75), (60, 77), (60, 153), (60, 305),
                                     (100, 36), (100, 37), (100, 74), (100, 75), (100, 76), (100, 77), (100, 152),
                                     (100, 153), (100, 305), (330, 153), (530, 16), (530, 37), (530, 75)])
def test_tiles(M, n, tiles):  # noqa: F811
    inst = _instance(n, n // 5, 0.2)
    P = 128 * tiles - 5
    _same(M, inst, I.normal_starts(inst, P, std=0.4, seed=P).Z0, M.PREC_BF16, T=4, period=2)


@pytest.mark.parametrize("tiles,period,prec,one_launch", [(78, 1, "PREC_BF16", False), (78, 2, "PREC_BF16", False),
                                                          (78, 1, "PREC_FP8", True), (120, 2, "PREC_BF16X1", True)])
def test_part_empty_waves(M, tiles, period, prec, one_launch):  # noqa: F811
    """d > 1024 beyond one wave: whichever kernels run, the same bits."""
    inst = _instance(1290, 258, 0.01)
    P = 128 * tiles - 3
    _same(M, inst, I.normal_starts(inst, P, std=0.3, seed=tiles).Z0, getattr(M, prec), one_launch, T=3, period=period)


@pytest.mark.parametrize("prec", ["PREC_BF16", "PREC_FP8"])
def test_many_steps(M, prec):  # noqa: F811
    inst = _instance(130, 26, 0.2)
    _same(M, inst, I.normal_starts(inst, 300, std=0.4, seed=8).Z0, getattr(M, prec), T=300, period=5)
