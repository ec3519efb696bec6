"""A tuned choice holds for its kind of call: one made for a general B or while
launch timing is on, where the streamed default runs step by step, does not take
a later identity-topped, untimed call of the shape off the one-launch kernel."""
import numpy as np
import pytest

from paper_2412_13576_gb300 import instances as I

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


def _run(M, inst, B, P, T):
    import torch
    ldc = M.round16(inst.n)
    Z = dev(I.normal_starts(inst, P, std=0.3, seed=2).Z0.astype(np.float32))
    Mm, V = torch.zeros_like(Z), torch.zeros_like(Z)
    cand = torch.zeros((P * (T + 1), ldc), dtype=torch.int8, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    flags = torch.zeros(1, dtype=torch.int32, device="cuda")
    M.extract(dev(B), dev((inst.u - inst.l).astype(np.int32)), Z, Mm, V, t0=0, T=T,
              cfg=M.default_config(precision=M.PREC_BF16 | M.PREC_AUTOTUNE), cand=cand, cand_count=cnt, flags=flags, ldc=ldc)
    torch.cuda.synchronize()


@pytest.mark.parametrize("n", [330, 400, 487, 600])
@pytest.mark.parametrize("first", ["general", "timed"])
def test_choice_of_another_kind(M, n, first):
    lib = M.lib()
    lib.mape_autotune_clear()
    inst = I.uneven_single(n)
    P, T = 1024, 40
    B = inst.B
    general = np.ascontiguousarray(B[np.r_[1:inst.d, 0, inst.d:n]])  # the identity's rows turned
    if first == "general":
        _run(M, inst, general, P, T)
    else:
        M.launch_timing(True)
        try:
            _run(M, inst, B, P, T)
        finally:
            M.launch_timing(False)
    _run(M, inst, B, P, T)  # tunes its own kind
    before = lib.mape_launch_count()
    _run(M, inst, B, P, T)
    assert lib.mape_launch_count() - before < T  # step by step: at least two launches a step
    info = M.autotune_info(n, inst.d, P, M.PREC_BF16)
    assert (info["path"], info["wF"], info["wG"]) == ("streamed", 256, 256)
    before = lib.mape_launch_count()
    _run(M, inst, general, P, T)
    _run(M, inst, general, P, T)
    assert lib.mape_launch_count() - before > 2 * T  # a general B stays with its kernels
