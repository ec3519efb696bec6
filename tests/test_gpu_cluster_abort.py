"""A call of the one-launch streamed extraction whose blocks have given up
from the start (time-out flag 16 set before it): every block meets its
barriers and leaves, nothing is collected and the state is as it was."""
import numpy as np
import pytest

from paper_2412_13576_gb300 import instances as I

from .gpu_common import dev
from .test_gpu_cluster import M, _instance  # noqa: F401  (M is the module fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,P", [(150, 30, 300), (1300, 1180, 130), (150, 30, 39 * 128)])
@pytest.mark.parametrize("prec", ["PREC_BF16", "PREC_FP8"])
def test_given_up_call_ends(M, n, m, P, prec):  # noqa: F811
    import torch
    inst = _instance(n, m, 0.1)
    Z0 = I.normal_starts(inst, P, std=0.4, seed=n).Z0.astype(np.float32)
    Z = dev(Z0)
    Mm, V = torch.full_like(Z, 0.25), torch.full_like(Z, 0.5)
    ldc = M.round16(n)
    cand = torch.zeros((P, ldc), dtype=torch.int8, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    flags = torch.full((1,), 16, dtype=torch.int32, device="cuda")
    pr = getattr(M, prec)
    cfg = M.default_config(precision=pr if pr == M.PREC_FP8 else pr | M.PREC_STREAMED)
    M.extract(dev(inst.B), dev((inst.u - inst.l).astype(np.int32)), Z, Mm, V, t0=0, T=9, cfg=cfg, cand=cand,
              cand_count=cnt, flags=flags, ldc=ldc)
    torch.cuda.synchronize()
    assert int(flags.item()) == 16 and int(cnt.item()) == 0
    assert np.array_equal(Z.cpu().numpy(), Z0)
    assert float(Mm.min()) == float(Mm.max()) == 0.25 and float(V.min()) == float(V.max()) == 0.5
