"""The one-launch streamed extraction keeps its operands in the caller's M, V
and Z while it runs: at any address of theirs, from one start to many (with the
operands in the workspace, in one, two and all three of the arrays), the state
comes out as from the step-by-step kernels, nothing beside the arrays changes,
and a call that refuses B leaves them as they are."""
import numpy as np
import pytest

from paper_2412_13576_gb300 import instances as I

from .gpu_common import dev
from .test_gpu_cluster import M, _instance  # noqa: F401  (M is the module fixture)

pytestmark = pytest.mark.gpu

PAD = 64  # floats beside each array


def _call(M, B, inst, start, prec, off, T, stepwise):
    import torch
    P, d = start[0].shape
    bufs, views = [], []
    for a in start:
        buf = torch.full((P * d + 2 * PAD,), -7.5, dtype=torch.float32, device="cuda")
        view = buf[PAD + off:PAD + off + P * d].view(P, d)
        view.copy_(dev(a))
        bufs.append(buf)
        views.append(view)
    ldc = M.round16(inst.n)
    cand = torch.zeros((P * (T + 1), ldc), dtype=torch.int8, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    flags = torch.zeros(1, dtype=torch.int32, device="cuda")
    nb = M.lib().mape_extract_workspace_bytes(inst.n, d, P, prec)
    ws = torch.full((nb + 4096,), 0x5a, dtype=torch.uint8, device="cuda")
    M.launch_timing(stepwise)
    try:
        M.extract(dev(B), dev((inst.u - inst.l).astype(np.int32)), *views, t0=0, T=T,
                  cfg=M.default_config(precision=prec), cand=cand, cand_count=cnt, flags=flags, ldc=ldc, workspace=ws[:nb])
        torch.cuda.synchronize()
    finally:
        M.launch_timing(False)
    for buf in bufs:
        b = buf.cpu().numpy()
        assert np.all(b[:PAD + off] == -7.5) and np.all(b[PAD + off + P * d:] == -7.5)
    assert bool((ws[nb:] == 0x5a).all())
    k = int(cnt.item())
    rows = cand[:k].cpu().numpy()
    return [v.cpu().numpy() for v in views], rows[np.lexsort(rows.T[::-1])] if k else rows, int(flags.item())


@pytest.mark.parametrize("n,m,P", [(60, 12, 1), (60, 12, 129), (150, 30, 130), (150, 30, 400), (150, 30, 1000),
                                   (41, 5, 1013), (670, 637, 300), (487, 97, 4996), (100, 20, 20000)])
@pytest.mark.parametrize("prec", ["PREC_BF16", "PREC_BF16X1", "PREC_FP8"])
@pytest.mark.parametrize("off", [0, 1, 3])
def test_operands_in_the_callers_arrays(M, n, m, P, prec, off):  # noqa: F811
    inst = _instance(n, m, 0.1)
    pr = getattr(M, prec)
    pr = pr if pr == M.PREC_FP8 else pr | M.PREC_STREAMED
    rng = np.random.default_rng(P)
    Z0 = I.normal_starts(inst, P, std=0.4, seed=P).Z0.astype(np.float32)
    start = (Z0, rng.standard_normal(Z0.shape).astype(np.float32), rng.random(Z0.shape).astype(np.float32))
    got = _call(M, inst.B, inst, start, pr, off, 3, False)
    want = _call(M, inst.B, inst, start, pr, off, 3, True)
    for a, b in zip(got[0], want[0]):
        assert np.array_equal(a, b)
    assert np.array_equal(got[1], want[1]) and got[2] == want[2]


def test_refused_basis_leaves_the_state(M):  # noqa: F811
    inst = _instance(150, 30, 0.1)
    B = inst.B.copy()
    B[inst.d, 3] = 257  # not exact in BF16: flag 8
    Z0 = I.normal_starts(inst, 500, std=0.4, seed=1).Z0.astype(np.float32)
    start = (Z0, Z0 + 1, Z0 * Z0)
    state, rows, flags = _call(M, B, inst, start, M.PREC_BF16 | M.PREC_STREAMED, 0, 3, False)
    assert flags & 8 and len(rows) == 0
    for a, b in zip(state, start):
        assert np.array_equal(a, b)
