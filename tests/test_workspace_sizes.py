"""The one-launch extraction asks for no more device memory than the
step-by-step kernels that it stands in for: workspaces and requests as large as
before it came, so that a memory cap that admitted a request still does."""
import ctypes

import pytest

from paper_2412_13576_gb300 import mape as M

# (n, d, P): workspace, and device bytes of a request with 4 starts and 100
# steps in BF16, of the step-by-step kernels alone
BEFORE = {
    (20, 15, 256): (8675328, 11003256),
    (41, 36, 1013): (9491456, 21926391),
    (487, 390, 4096): (38196736, 534095569),
    (487, 390, 65536): (466556416, 5694321817),
    (50, 40, 65536): (77358080, 1618638470),
    (670, 33, 4236): (21380096, 707254158),
    (1000, 800, 4096): (66790912, 1052540536),
    (1300, 120, 4096): (32344576, 1302853632),
    (2000, 1600, 65536): (1689896448, 7852559362),
    (4000, 3200, 4096): (284881408, 4256806328),
}


@pytest.mark.parametrize("shape", list(BEFORE))
def test_no_larger_than_before(shape):
    lib = M.lib(build_if_missing=True)
    n, d, P = shape
    for prec in (M.PREC_BF16, M.PREC_BF16X1, M.PREC_FP8, M.PREC_BF16 | M.PREC_STREAMED):
        assert lib.mape_extract_workspace_bytes(n, d, P, prec) <= BEFORE[shape][0]
    cfg = M.default_config(T=100, precision=M.PREC_BF16)
    assert lib.mape_request_bytes(n, n - d, P, 4, ctypes.byref(cfg)) <= BEFORE[shape][1]
