"""The scoring pass's unit-step test (room left in the box against four entries
at a time) and its queue of remaining directions, against a numpy restatement
of Algorithm 1: rooms on both sides of the int8 range, entries -128 and 127,
few and all directions remaining, counts around a block of 256 and n around the
16-byte pieces and past the n that has the pre-pass.  Integers: equal."""
import numpy as np
import pytest

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


def _best(G, a, r, x, l, u):
    """(Delta f, k, e < 0, lambda) of the best move (w = 0), or None."""
    best = None
    for neg in (0, 1):
        g = -G if neg else G
        room = np.where(g > 0, u - x, x - l)
        lam = np.where(g != 0, room // np.maximum(np.abs(g), 1), 1 << 20).min(axis=1)
        b = g @ r
        for k in np.nonzero((lam >= 1) & (lam <= 255))[0]:
            t = np.arange(1, lam[k] + 1)
            df = t * t * a[k] + t * b[k]
            j = int(df.argmin())
            c = (int(df[j]), int(k), neg, int(t[j]))
            best = c if best is None or c < best else best
    return best


@pytest.mark.parametrize("lanes", [1, 4, 32])
@pytest.mark.parametrize("n,K,kind", [(1, 3, "few"), (15, 257, "all"), (16, 600, "all"), (17, 255, "extreme"),
                                      (33, 1500, "few"), (130, 513, "extreme"), (936, 300, "few"), (1212, 40, "few"),
                                      (4097, 300, "few")])
def test_unit_steps_and_queue(M, n, K, kind, lanes):
    rng = np.random.default_rng(n * 7 + K)
    span = 255 if kind == "extreme" else 3
    l = rng.integers(-100, 1, size=n)
    u = l + rng.integers(span // 2, span + 1, size=n)
    x0 = rng.integers(l, u + 1, size=(3, n))
    if kind == "extreme":    # rooms of 126 .. 129 with entries at the ends of int8, one or two a row
        l, u = np.full(n, -129), np.full(n, 126)
        x0 = rng.integers(-3, 2, size=(3, n))
    G = np.zeros((K, n), np.int64)
    for k in range(K):
        cols = rng.choice(n, size=min(n, 2 if kind == "extreme" else 1 + k % 3), replace=False)
        G[k, cols] = rng.choice([-128, -127, -126, 126, 127] if kind == "extreme" else [-2, -1, 1, 2], size=len(cols))
    if kind == "few":        # most rows cannot step either way
        full = rng.random(K) < 0.9
        G[full] = 4 * rng.choice([-1, 1], size=(int(full.sum()), n))
    qd = rng.integers(0, 3, size=n)
    c = rng.integers(-40, 41, size=n)
    a = (G * G) @ qd
    buf = np.zeros((K, M.round16(n)), np.int8)
    buf[:, :n] = G
    idx = np.arange(n, dtype=np.int32)
    X = dev(x0.astype(np.int32))
    fval, iters, moves, nmoves = M.augment_run(dev(buf), n, dev(a), dev(np.zeros(K, np.int64)), dev(idx), dev(idx),
                                               dev(qd.astype(np.int32)), dev(c.astype(np.int32)), None,
                                               dev(l.astype(np.int32)), dev(u.astype(np.int32)), X, max_iters=6,
                                               moves_cap=8, lanes=lanes)
    moves, nmoves = moves.cpu().numpy(), nmoves.cpu().numpy()
    total = 0
    for s in range(3):
        x = x0[s].copy()
        want = []
        for _ in range(6):
            m = _best(G, a, 2 * qd * x + c, x, l, u)
            if m is None or m[0] >= 0:
                break
            x = x + (-1 if m[2] else 1) * m[3] * G[m[1]]
            want.append((m[1], -1 if m[2] else 1, m[3], int(qd @ (x * x) + c @ x)))
        assert [tuple(int(v) for v in moves[s, i]) for i in range(nmoves[s])] == want
        assert np.array_equal(X[s].cpu().numpy(), x) and int(fval[s].item()) == int(qd @ (x * x) + c @ x)
        total += len(want)
    assert n == 1 or total > 0
