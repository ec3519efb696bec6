"""A handle whose allocator has no block for a whole stage takes its buffers one
by one: the same directions and point as with one block, and everything is given
back; where a single buffer does not fit either, the stage is refused and the
handle goes on with what fits."""
import ctypes as C

import numpy as np
import pytest

from paper_2412_13576_gb300 import instances as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2412_13576_gb300 import mape
    mape.lib(build_if_missing=True)
    return mape


class Allocator:
    """torch's caching allocator, refusing requests above `limit`."""

    def __init__(self, M, limit=None):
        import torch
        self.limit, self.sizes, self.refused, self.held = limit, [], 0, {}

        def alloc(nbytes, stream, ctx):
            if self.limit is not None and nbytes > self.limit:
                self.refused += 1
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), stream=int(stream or 0))
            self.sizes.append(nbytes)
            self.held[p] = nbytes
            return p

        def free(ptr, nbytes, stream, ctx):
            assert self.held.pop(ptr) == nbytes
            torch.cuda.caching_allocator_delete(int(ptr))

        self.fns = (M._ALLOC_FN(alloc), M._FREE_FN(free))
        self.M = M

    def __enter__(self):
        f = self.fns
        self.M.lib().mape_set_allocator(C.cast(f[0], C.c_void_p), C.cast(f[1], C.c_void_p), None)
        return self

    def __exit__(self, *exc):
        self.M.lib().mape_set_allocator(None, None, None)


CAP = 20000  # candidate rows of a handle


def _solve(M, inst, P):
    cfg = M.default_config(T=12, precision=M.PREC_BF16, cand_capacity=CAP)
    with M.Instance.from_generated(inst, cfg) as h:
        h.extract_directions(P, G0=I.uniform_samples(inst, P, 3).G0)
        h.wait(60)
        h.augment(inst.xbar[None, :])
        h.wait(60)
        return h.directions(), h.solution()


def test_buffers_one_by_one(M):
    inst = I.uneven_single(120)
    P = 700
    with Allocator(M) as whole:
        want = _solve(M, inst, P)
    assert not whole.held and whole.refused == 0
    # a little above the largest single buffer, the stage's work space
    lib, ldg = M.lib(), M.round16(inst.n)
    work = max(lib.mape_extract_workspace_bytes(inst.n, inst.d, P, M.PREC_BF16), lib.mape_dedup_workspace_bytes(CAP, ldg),
               lib.mape_minimal_workspace_bytes(CAP, inst.n))
    assert max(whole.sizes) > 1.2 * work
    with Allocator(M, limit=work + 4096) as parts:
        got = _solve(M, inst, P)
    assert parts.refused > 0 and not parts.held
    assert np.array_equal(got[0], want[0]) and got[0].shape[0] > 0
    assert np.array_equal(got[1][0], want[1][0]) and got[1][1] == want[1][1]


def test_a_buffer_too_large(M):
    inst = I.uneven_single(120)
    cfg = M.default_config(T=12, precision=M.PREC_BF16)
    with Allocator(M) as a:
        with M.Instance.from_generated(inst, cfg) as h:
            a.limit = 100 << 10
            with pytest.raises(M.MapeError) as e:
                h.extract_directions(700, Z0=I.normal_starts(inst, 700, std=0.4, seed=1).Z0)
            assert e.value.code == -11 and a.refused > 1
            a.limit = None
            h.extract_directions(64, Z0=I.normal_starts(inst, 64, std=0.4, seed=1).Z0)
            h.wait(60)
            assert h.directions().shape[0] > 0
    assert not a.held
