"""What goes wrong between a request's extraction and Algorithm 1, on the thread
that takes it there: a start that is not feasible fails its request alone, its
slot and memory are free for the next, the others' results are theirs.  And the
streams that closed handles leave to new ones: several threads at once, with the
idle ones destroyed in between."""
import threading

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


@pytest.mark.parametrize("keep", [False, True])
@pytest.mark.parametrize("batch", [False, True])
def test_infeasible_start(M, keep, batch):
    insts = [I.uneven_single(n) for n in (40, 60, 150, 320)]
    cfg = M.default_config(T=30, precision=M.PREC_BF16)
    starts = [I.normal_starts(x, 256, std=0.4, seed=k).Z0 for k, x in enumerate(insts)]

    def bad_start(x):
        X0 = x.xbar.copy()
        X0[x.d] += 1 if X0[x.d] < x.u[x.d] else -1
        return X0

    with M.Server(cfg, mem_cap_bytes=32 << 30, max_slots=2, keep_directions=keep, batch_extraction=batch) as srv:
        if batch:  # a batch of starts is refused as a whole: the requests one after the other
            for x, Z0 in zip(insts, starts):
                bad = srv.submit(x, 256, Z0=Z0, X0=bad_start(x))
                srv.wait_all(120)
                assert srv.info(bad)["state"] == "FAILED" and srv.info(bad)["error"] == -5
                srv.release(bad)
        ids = []
        for k, (x, Z0) in enumerate(zip(insts, starts)):
            ids.append(srv.submit(x, 256, Z0=Z0))
            if not batch:
                ids.append(srv.submit(x, 256, Z0=Z0, X0=bad_start(x)))
        srv.wait_all(120)
        stats = srv.stats()
        assert stats["failed"] == len(insts) and stats["completed"] == len(insts)
        assert stats["running"] == 0 and stats["mem_in_use"] == 0
        good = ids if batch else ids[::2]
        for i in ids:
            info = srv.info(i)
            assert (info["state"] == "DONE") == (i in good) and info["error"] == (0 if i in good else -5)
        for i, x, Z0 in zip(good, insts, starts):
            with M.Instance.from_generated(x, cfg) as h:
                h.extract_directions(256, Z0=Z0)
                h.wait(60)
                h.augment(x.xbar[None, :])
                h.wait(60)
                want = h.solution()
            got = srv.result(i)
            assert np.array_equal(got[0], want[0]) and got[1] == want[1]


def test_streams_of_closed_handles(M):
    inst = I.uneven_single(50)
    cfg = M.default_config(T=10, precision=M.PREC_BF16)
    Z0 = I.normal_starts(inst, 128, std=0.4, seed=1).Z0

    def solve():
        with M.Instance.from_generated(inst, cfg) as h:
            h.extract_directions(128, Z0=Z0)
            h.wait(60)
            return h.directions()

    want = solve()
    wrong, stop = [], threading.Event()

    def work():
        for _ in range(12):
            try:
                if not np.array_equal(solve(), want):
                    wrong.append("directions")
            except Exception as e:
                wrong.append(repr(e))

    def trim():
        while not stop.wait(0.01):
            M.trim_memory()

    threads = [threading.Thread(target=work) for _ in range(4)]
    side = threading.Thread(target=trim)
    for t in threads + [side]:
        t.start()
    for t in threads:
        t.join(120)
    stop.set()
    side.join(60)
    assert not wrong and not any(t.is_alive() for t in threads + [side])
