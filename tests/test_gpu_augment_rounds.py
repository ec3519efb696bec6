"""The scoring pass of Algorithm 1 where a block takes several rounds of
directions: the queue carried from round to round and emptied several times,
rounds handed out one by one, and passes that change between the two forms
because the share of directions with room is not what the sample or the pass
before said.  Against a numpy restatement of Algorithm 1; integers: equal."""
import numpy as np
import pytest

from .gpu_common import dev
from .test_gpu_augment_room import M, _best  # noqa: F401  (M is the module fixture)

pytestmark = pytest.mark.gpu

S = 304  # eight blocks a start


def _rows(rng, K, n, share, sample):
    """K directions of which `share` have room on rooms of 2 .. 4 (entries of
    1 or 2, the others' 6); `sample`: what the 32 rows that are looked at first
    are instead."""
    G = np.zeros((K, n), np.int64)
    has = rng.random(K) < share
    if sample is not None:
        has[(np.arange(32) * K) >> 5] = sample
    for k in range(K):
        cols = rng.choice(n, size=min(n, 3), replace=False)
        G[k, cols] = rng.choice([-1, 1], size=len(cols)) * (1 + k % 2 if has[k] else 6)
    return G


@pytest.mark.parametrize("lanes,K,n", [(1, 9000, 16), (1, 9216, 33), (8, 2600, 50), (32, 1500, 20), (32, 500, 300)])
@pytest.mark.parametrize("share,sample", [(0.1, None), (0.1, True), (0.6, None), (0.6, False), (1.0, None), (0.0, True)])
@pytest.mark.parametrize("quartic", [False, True])
def test_rounds(M, lanes, K, n, share, sample, quartic):  # noqa: F811
    rng = np.random.default_rng(K + n + int(10 * share))
    l = -rng.integers(2, 5, size=n)
    u = rng.integers(2, 5, size=n)
    x0 = np.clip(rng.integers(-1, 2, size=(S, n)), l, u)
    G = _rows(rng, K, n, share, sample)
    qd = rng.integers(0, 3, size=n)
    c = rng.integers(-40, 41, size=n)
    w = np.zeros(n, np.int64)  # the quartic kernel with a term that is 0: the same moves
    a, q4 = (G * G) @ qd, (G ** 4) @ w
    buf = np.zeros((K, M.round16(n)), np.int8)
    buf[:, :n] = G
    idx = np.arange(n, dtype=np.int32)
    X = dev(x0.astype(np.int32))
    iters = 4
    fval, _, moves, nmoves = M.augment_run(dev(buf), n, dev(a), dev(q4), dev(idx), dev(idx), dev(qd.astype(np.int32)),
                                           dev(c.astype(np.int32)), dev(w.astype(np.int32)) if quartic else None,
                                           dev(l.astype(np.int32)), dev(u.astype(np.int32)), X, max_iters=iters,
                                           moves_cap=iters, lanes=lanes)
    moves, nmoves, X, fval = (t.cpu().numpy() for t in (moves, nmoves, X, fval))
    total = 0
    for s in (0, 1, 77, 152, 303):
        x = x0[s].copy()
        want = []
        for _ in range(iters):
            m = _best(G, a, 2 * qd * x + c, x, l, u)
            if m is None or m[0] >= 0:
                break
            x = x + (-1 if m[2] else 1) * m[3] * G[m[1]]
            want.append((m[1], -1 if m[2] else 1, m[3], int(qd @ (x * x) + c @ x)))
        assert [tuple(int(v) for v in moves[s, i]) for i in range(nmoves[s])] == want
        assert np.array_equal(X[s], x) and int(fval[s]) == int(qd @ (x * x) + c @ x)
        total += len(want)
    assert total > 0
