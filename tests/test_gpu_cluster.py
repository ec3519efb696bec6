"""The one-launch streamed extraction (a cluster of blocks per tile of 128
starts) against the step-by-step streamed kernels, which run while launch
timing is on: the same Adam state bit for bit, the same candidates, the same
gradient.  The step-by-step kernels are the ones the per-step oracle cases of
test_gpu_streamed.py were written for; shapes here sit at the edges of the
cluster path's slices, chunks and accumulator blocks."""
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


def _instance(n, m, dens=0.1):
    return I.make_instance(f"edge_n{n}_m{m}", n, m, c_k=3, c_density=dens, lo=-5, hi=5, q_k=3, q_density=0.1,
                           lin_k=10, seed=100 * n + m)


def _run(M, inst, Z0, prec, *, T, t0=0, period=1, eps=1e-8, moments=None, stepwise=False):
    import torch
    P = Z0.shape[0]
    ldc = M.round16(inst.n)
    Z = dev(Z0.astype(np.float32))
    Mm, V = (torch.zeros_like(Z), torch.zeros_like(Z)) if moments is None else tuple(dev(a) for a in moments)
    cand = torch.zeros((P * (T + 1), ldc), dtype=torch.int8, device="cuda")
    cnt = torch.zeros(1, dtype=torch.int64, device="cuda")
    flags = torch.zeros(1, dtype=torch.int32, device="cuda")
    phi = torch.zeros(P, dtype=torch.float32, device="cuda")
    grad = torch.zeros_like(Z)
    cfg = M.default_config(precision=prec | M.PREC_STREAMED if prec != M.PREC_FP8 else prec, period=period)
    cfg.eps = eps
    M.launch_timing(stepwise)
    try:
        before = M.lib().mape_launch_count()
        M.extract(dev(inst.B), dev((inst.u - inst.l).astype(np.int32)), Z, Mm, V, t0=t0, T=T, cfg=cfg, cand=cand,
                  cand_count=cnt, flags=flags, ldc=ldc, dbg_phi=phi, dbg_grad=grad)
        torch.cuda.synchronize()
        launches = M.lib().mape_launch_count() - before
    finally:
        M.launch_timing(False)
    k = int(cnt.item())
    rows = cand[:k].cpu().numpy()
    rows = rows[np.lexsort(rows.T[::-1])] if k else rows
    return dict(Z=Z.cpu().numpy(), M=Mm.cpu().numpy(), V=V.cpu().numpy(), flags=int(flags.item()), rows=rows,
                grad=grad.cpu().numpy(), phi=phi.cpu().numpy(), launches=launches)


def _same(M, inst, Z0, prec, **kw):
    a = _run(M, inst, Z0, prec, **kw)
    b = _run(M, inst, Z0, prec, stepwise=True, **kw)
    assert a["launches"] < b["launches"] or kw["T"] < 2  # the two routes did run
    for k in ("Z", "M", "V", "grad"):
        assert np.array_equal(a[k], b[k], equal_nan=True), k
    assert a["flags"] == b["flags"]
    assert np.array_equal(a["rows"], b["rows"])
    # Phi is summed by atomics in another order: n + d terms of at most the total
    fin = np.isfinite(b["phi"])
    assert np.array_equal(fin, np.isfinite(a["phi"]))
    assert np.all(np.abs(a["phi"][fin] - b["phi"][fin]) <= (inst.n + inst.d) * 2.0 ** -23 * np.abs(b["phi"][fin]) + 1e-6)
    return a


# slices of less than one 16-wide unit per block, odd d, d and rows at the
# 16 / 32 / 64 edges, more than 128 rows or 256 coordinates per block
SHAPES = [(20, 5, 0.5), (17, 1, 0.5), (33, 1, 0.5), (64, 32, 0.3), (129, 33, 0.2), (160, 64, 0.2), (487, 97, 0.1),
          (777, 155, 0.1), (1300, 1180, 0.02), (2600, 300, 0.02)]


@pytest.mark.parametrize("n,m,dens", SHAPES)
@pytest.mark.parametrize("prec", ["PREC_BF16", "PREC_BF16X1", "PREC_FP8"])
def test_shapes(M, n, m, dens, prec):
    inst = _instance(n, m, dens)
    Z0 = I.normal_starts(inst, 130, std=0.3, seed=n).Z0
    r = _same(M, inst, Z0, getattr(M, prec), T=6)
    if n <= 160:
        assert r["rows"].shape[0] > 0


@pytest.mark.parametrize("P", [1, 127, 128, 129, 38 * 128, 38 * 128 + 1])
def test_starts(M, P):
    """Ragged tiles, and both sides of the cluster-size rule (38 tiles)."""
    inst = _instance(150, 30, 0.2)
    _same(M, inst, I.normal_starts(inst, P, std=0.4, seed=P).Z0, M.PREC_BF16, T=5)


@pytest.mark.parametrize("t0,T,period", [(0, 1, 1), (3, 7, 2), (5, 9, 3), (0, 8, 8), (7, 4, 50)])
@pytest.mark.parametrize("prec", ["PREC_BF16", "PREC_FP8"])
def test_periods_and_continued_runs(M, t0, T, period, prec):
    inst = _instance(200, 40, 0.1)
    st = I.normal_starts(inst, 200, std=0.4, seed=5).Z0
    rng = np.random.default_rng(9)
    mom = (rng.standard_normal(st.shape).astype(np.float32), rng.random(st.shape).astype(np.float32))
    _same(M, inst, st, getattr(M, prec), T=T, t0=t0, period=period, moments=mom)


@pytest.mark.parametrize("eps", [1e-8, 1e-20])
@pytest.mark.parametrize("prec", ["PREC_BF16", "PREC_FP8"])
def test_values_at_the_edges(M, prec, eps):
    """Zero starts, exact ties, subnormal and huge coordinates, starts on both
    sides of ||z||_inf = 1 and of a power of two (FP8 scales), infinities and
    NaN; an epsilon below the range of the fast second-moment form."""
    inst = _instance(100, 20, 0.2)
    rng = np.random.default_rng(3)
    Z0 = (rng.standard_normal((140, inst.d)) * 0.5).astype(np.float32)
    Z0[0] = 0.0
    Z0[1] = 0.5
    Z0[2] = np.where(np.arange(inst.d) % 2 == 0, 1.5, -2.5)
    Z0[3] = 1e-40
    Z0[4, :7] = [3e6, -5e6, 4194304.0, 8388609.0, 1e20, -0.0, 2097152.5]
    Z0[5] = np.clip(Z0[5], -0.9, 0.9)
    Z0[5, 3] = Z0[5, 9] = 0.95
    Z0[6] *= 7.9999 / np.abs(Z0[6]).max()
    Z0[7, 2] = np.inf
    Z0[8, 2] = np.nan
    _same(M, inst, Z0, getattr(M, prec), T=8, eps=eps)
