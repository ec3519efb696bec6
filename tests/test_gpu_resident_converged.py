"""The resident and the step-by-step kernels with their debug outputs on, which
their lanes write one by one between the tensor-memory loads: the gradient and
the state of every start are those of its own small call, on a full chip, call
after call."""
import numpy as np
import pytest

from paper_2412_13576_gb300 import instances as I

from .gpu_common import dev
from .test_gpu_cluster import M, _instance  # noqa: F401  (M is the module fixture)

pytestmark = pytest.mark.gpu


def _run(M, inst, Z0, prec, T, stepwise):
    import torch
    P = Z0.shape[0]
    Z = dev(Z0)
    Mm, V, grad = torch.zeros_like(Z), torch.zeros_like(Z), torch.zeros_like(Z)
    phi = torch.zeros(P, dtype=torch.float32, device="cuda")
    ldc = M.round16(inst.n)
    cand = torch.zeros((P * (T + 1), ldc), dtype=torch.int8, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    flags = torch.zeros(1, dtype=torch.int32, device="cuda")
    M.launch_timing(stepwise)
    try:
        M.extract(dev(inst.B), dev((inst.u - inst.l).astype(np.int32)), Z, Mm, V, t0=0, T=T,
                  cfg=M.default_config(precision=prec), cand=cand, cand_count=cnt, flags=flags, ldc=ldc, dbg_phi=phi,
                  dbg_grad=grad)
        torch.cuda.synchronize()
    finally:
        M.launch_timing(False)
    return [t.cpu().numpy() for t in (grad, Z, Mm, V)]


@pytest.mark.parametrize("n,m,prec,stepwise", [(200, 40, "PREC_BF16", False), (20, 5, "PREC_BF16", False),
                                               (200, 40, "PREC_BF16X1", False), (487, 97, "PREC_BF16", True),
                                               (487, 97, "PREC_FP8", True)])
def test_every_start_as_alone(M, n, m, prec, stepwise):  # noqa: F811
    inst = _instance(n, m, 0.1)
    P, T = 24000, 2
    Z0 = I.normal_starts(inst, P, std=0.4, seed=n).Z0.astype(np.float32)
    pr = getattr(M, prec)
    at = np.r_[0:128, 9088:9216, P - 40:P]
    want = _run(M, inst, np.ascontiguousarray(Z0[at]), pr, T, stepwise)
    first = _run(M, inst, Z0, pr, T, stepwise)
    for a, b in zip(first, want):
        assert np.array_equal(a[at], b)
    for _ in range(3):
        for a, b in zip(_run(M, inst, Z0, pr, T, stepwise), first):
            assert np.array_equal(a, b)
