"""The work that a user of this framework has it do, as cases to be timed and
compared: the stages of the path through their public entry points
(paper_2412_13576_gb300.mape) and two whole calls (an instance handle, a
request server).  Shapes are those of the five workloads of
paper_2412_13576_gb300.instances and of ragged sizes between them.

A case is a dict with "kind" (one of the functions below) and its sizes:

  extract   Algorithm 2 for one instance: T Adam steps of P starts, then the
            set union of what was collected
  batch     the same for several uneven instances in one batched call
  project   starting points z0 = (B^T B)^{-1} B^T g
  filter    candidate rows -> distinct rows -> kernel test -> minimality
            filter -> coefficients of Algorithm 1
  augment   Algorithm 1 from S starts with K directions
  initial   feasible points by Eq. (4)
  handle    one instance through its handle, from host arrays to host arrays
  serve     several uneven requests through a request server
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2412_13576_gb300 import instances as I
from paper_2412_13576_gb300 import mape

DEV = "cuda"


def listed():
    return [
        # the smallest call: the 20-variable workload with all its starts and
        # steps; launches, copies and waits are most of it
        dict(name="extract_small", kind="extract", family="small", n=20, P=256, T=200, period=1, prec="bf16", std=2.0),
        # the medium workload's extraction (B and the state fit on chip)
        dict(name="extract_medium", kind="extract", family="medium", n=200, P=8192, T=250, period=1, prec="bf16",
             std=0.8),
        # a request of the serving mix that does not fit on chip: odd n, the
        # mix's own P
        dict(name="extract_uneven", kind="extract", family="uneven", n=487, P=4096, T=100, period=1, prec="bf16",
             std=0.4),
        # the large workload in its stated precision, with all its starts,
        # from its own distribution, between two collections
        dict(name="extract_large", kind="extract", family="large", n=2000, P=65536, T=50, period=50, prec="fp8",
             std=2.0),
        # uneven instances that arrive together, as the batched workload has them
        dict(name="batch_uneven", kind="batch", n_lo=50, n_hi=1000, count=12, P=1024, T=50, std=0.4),
        # the starts of a request of the upper half of the serving mix
        dict(name="project_uneven", kind="project", family="uneven", n=1000, P=4096),
        # everything after the extraction up to Algorithm 1, at the number of
        # candidates that a pass of the medium and of the large workload leaves
        dict(name="filter_medium", kind="filter", family="medium", n=200, K=120000),
        dict(name="filter_large", kind="filter", family="large", n=2000, K=300000),
        # multi-start augmentation with a set of the medium workload's size
        dict(name="augment_medium", kind="augment", family="medium", n=200, K=60000, S=64, iters=400),
        # initial feasible points for the medium workload
        dict(name="initial_medium", kind="initial", family="medium", n=200, P=1024, T=200),
        # the medium workload as its user runs it: host arrays in, the
        # direction set and the best point out
        dict(name="handle_medium", kind="handle", family="medium", n=200, P=8192, T=1000),
        # requests of the serving mix admitted together
        dict(name="serve_uneven", kind="serve", n_lo=30, n_hi=1500, count=16, P=4096, T=100, std=0.4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["extract", "extract", "extract", "extract", "batch", "project", "filter", "filter", "augment",
                       "initial", "handle", "serve"])
    if kind == "extract":
        n = _log_int(rng, 20, 2400)
        P = _log_int(rng, 100, 16384)
        T = max(10, min(_log_int(rng, 20, 400), int(4e9 / (n * P))))
        prec = rng.choice(["bf16", "bf16", "fp8", "bf16x1"])
        return dict(kind=kind, family="uneven", n=n, P=P, T=T, period=rng.choice([1, 1, 7, 50]), prec=prec,
                    std=rng.choice([0.3, 0.6, 2.0]))
    if kind == "batch":
        return dict(kind=kind, n_lo=rng.randint(30, 100), n_hi=rng.randint(300, 1100), count=rng.randint(3, 16),
                    P=_log_int(rng, 200, 3000), T=rng.randint(15, 60), std=rng.choice([0.3, 0.6]))
    if kind == "project":
        return dict(kind=kind, family="uneven", n=_log_int(rng, 20, 1200), P=_log_int(rng, 100, 12000))
    if kind == "filter":
        n = _log_int(rng, 20, 2000)
        return dict(kind=kind, family="uneven", n=n, K=_log_int(rng, 500, 100000))
    if kind == "augment":
        return dict(kind=kind, family=rng.choice(["uneven", "large"]), n=_log_int(rng, 20, 1000),
                    K=_log_int(rng, 500, 50000), S=_log_int(rng, 1, 64), iters=rng.randint(20, 300))
    if kind == "initial":
        return dict(kind=kind, family="uneven", n=_log_int(rng, 20, 400), P=_log_int(rng, 64, 2048),
                    T=rng.randint(20, 200))
    if kind == "handle":
        return dict(kind=kind, family="uneven", n=_log_int(rng, 20, 600), P=_log_int(rng, 200, 2500),
                    T=rng.randint(50, 100))
    return dict(kind=kind, n_lo=30, n_hi=rng.randint(200, 1200), count=rng.randint(4, 16), P=_log_int(rng, 256, 4096),
                T=rng.randint(20, 100), std=rng.choice([0.3, 0.6]))


# ---------------------------------------------------------------------------
# inputs

def _instance(family, n, seed):
    """An instance of a workload's family at n variables (m as the workload has it)."""
    if family == "small":
        return I.make_instance("small", n, max(1, n // 4), c_k=2, c_density=None, lo=-5, hi=5, q_k=3, q_density=0.3,
                               lin_k=10, seed=seed)
    if family == "medium":
        return I.make_instance("medium", n, max(1, n // 5), c_k=3, c_density=0.1, lo=0, hi=10, q_k=5, q_density=0.05,
                               lin_k=20, seed=seed)
    if family == "large":
        return I.make_instance("large", n, max(1, n // 5), c_k=5, c_density=0.01, lo=-20, hi=20, q_k=5,
                               q_density=0.005, lin_k=20, w_max=3, seed=seed)
    return I.make_instance("uneven", n, max(1, n // 5), c_k=3, c_density=0.1, lo=-5, hi=5, q_k=3, q_density=0.3,
                           lin_k=10, seed=seed)


def _uneven_instances(case, seed):
    """`count` instances with n log-spaced over [n_lo, n_hi], densities 0.05 to 0.2."""
    rng = np.random.default_rng(seed)
    lo, hi, k = case["n_lo"], case["n_hi"], case["count"]
    out = []
    for i in range(k):
        n = int(round(lo * (hi / lo) ** (i / max(1, k - 1))))
        out.append(I.make_instance(f"uneven_{i}", n, max(1, n // 5), c_k=3, c_density=float(rng.uniform(0.05, 0.2)),
                                   lo=-5, hi=5, q_k=3, q_density=0.3, lin_k=10, seed=seed * 100 + i))
    return out


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 7919 + 11)
    return g


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to(DEV)


def _span(inst):
    return _dev((inst.u - inst.l).astype(np.int32))


PREC = {"bf16": mape.PREC_BF16, "bf16x1": mape.PREC_BF16X1, "fp8": mape.PREC_FP8}


def _call_state(inst, P, T, period, std, g, cfg):
    """One extraction's buffers: starts, state, candidate rows and counters, and
    the program's own buffer of directions (rows beyond their number stay 0)."""
    d, ldc = inst.d, mape.round16(inst.n)
    rows = P * (T // period + 1)  # one per start and collection: none is ever dropped
    Z0 = torch.randn((P, d), generator=g, device=DEV) * std
    nb = mape.lib().mape_extract_workspace_bytes(inst.n, d, P, cfg.precision)
    return dict(B=_dev(inst.B), span=_span(inst), Z0=Z0, Z=torch.empty_like(Z0), M=torch.empty_like(Z0),
                V=torch.empty_like(Z0), kept=torch.zeros((rows, ldc), dtype=torch.int8, device=DEV),
                cand=torch.empty((rows, ldc), dtype=torch.int8, device=DEV),
                cand_count=torch.zeros(1, dtype=torch.int64, device=DEV),
                flags=torch.zeros(1, dtype=torch.int32, device=DEV), ldc=ldc, n=inst.n,
                workspace=torch.empty(max(int(nb), 16), dtype=torch.uint8, device=DEV))


def _kernel_rows(inst, K, seed):
    """K candidate rows g = B z in canonical sign (int8, pitch round16(n)):
    integer z of mixed lengths, with about a quarter of the rows repeated, as
    the starts of an extraction collect one direction more than once."""
    g = _gen(seed)
    n, d, ldc = inst.n, inst.d, mape.round16(inst.n)
    Bm = _dev(inst.B[d:]).float()
    uniq = max(1, (3 * K) // 4)
    out = torch.zeros((K, ldc), dtype=torch.int8, device=DEV)
    std = torch.tensor([0.25, 0.35, 0.5, 0.6], device=DEV)
    for a in range(0, uniq, 65536):
        k = min(65536, uniq - a)
        s = std[torch.randint(0, 4, (k, 1), generator=g, device=DEV)]
        z = (torch.randn((k, d), generator=g, device=DEV) * s).round_().clamp_(-6, 6)
        one = torch.randint(0, d, (k,), generator=g, device=DEV)
        z[torch.arange(k, device=DEV), one] += (z.abs().sum(1) == 0).float()
        v = torch.cat([z, z @ Bm.T], dim=1)
        v = v * (v.abs().amax(1, keepdim=True) <= 127)  # a row that does not fit in int8 becomes the unit row below
        dead = v.abs().sum(1) == 0
        v[dead, :d] = 0.0
        first = (v != 0).float().argmax(1)
        sg = torch.sign(v[torch.arange(k, device=DEV), first])
        out[a:a + k, :n] = (v * sg[:, None]).to(torch.int8)
        if bool(dead.any()):  # B e_j for some j: a kernel element of small entries
            j = torch.randint(0, d, (int(dead.sum()),), generator=g, device=DEV)
            e = torch.zeros((j.numel(), d), device=DEV)
            e[torch.arange(j.numel(), device=DEV), j] = 1.0
            rows = torch.zeros((j.numel(), ldc), dtype=torch.int8, device=DEV)
            rows[:, :n] = torch.cat([e, e @ Bm.T], dim=1).to(torch.int8)
            out[a:a + k][dead] = rows
    if K > uniq:
        out[uniq:] = out[torch.randint(0, uniq, (K - uniq,), generator=g, device=DEV)]
    return out[torch.randperm(K, generator=g, device=DEV)].contiguous()


def _problem(inst):
    qr, qc, qv = (_dev(x) for x in mape.coo_upper(inst.Q))
    return dict(qr=qr, qc=qc, qv=qv, c=_dev(inst.c), w=None if inst.w is None else _dev(inst.w), l=_dev(inst.l),
                u=_dev(inst.u))


def prepare(case, seed):
    kind = case["kind"]
    g = _gen(seed)
    if kind == "extract":
        inst = _instance(case["family"], case["n"], seed)
        cfg = mape.default_config(T=case["T"], period=case["period"], precision=PREC[case["prec"]])
        return dict(kind=kind, cfg=cfg, call=_call_state(inst, case["P"], case["T"], case["period"], case["std"], g, cfg))
    if kind == "batch":
        cfg = mape.default_config(T=case["T"], precision=mape.PREC_BF16)
        calls = [_call_state(x, case["P"] * (4 if i % 3 == 2 else 1), case["T"], 1, case["std"], g, cfg)
                 for i, x in enumerate(_uneven_instances(case, seed))]
        return dict(kind=kind, cfg=cfg, calls=calls)
    if kind == "project":
        inst = _instance(case["family"], case["n"], seed)
        span = _span(inst).float()
        G0 = (torch.rand((case["P"], inst.n), generator=g, device=DEV) * 2 - 1) * span
        return dict(kind=kind, B=_dev(inst.B), G0=G0)
    if kind == "filter":
        inst = _instance(case["family"], case["n"], seed)
        K, ldg = case["K"], mape.round16(inst.n)
        zeros = lambda shape, dt: torch.zeros(shape, dtype=dt, device=DEV)  # noqa: E731
        return dict(kind=kind, n=inst.n, A=_dev(inst.A), cand=_kernel_rows(inst, K, seed),
                    ok=zeros(K, torch.uint8), keep=zeros(K, torch.uint8), rows=zeros((K, ldg), torch.int8),
                    a=zeros(K, torch.int64), q4=zeros(K, torch.int64), **_problem(inst))
    if kind == "augment":
        inst = _instance(case["family"], case["n"], seed)
        p = _problem(inst)
        G = mape.dedup(_kernel_rows(inst, case["K"], seed), case["K"], inst.n)
        G = torch.cat([G])  # its own memory, as a kept set has
        a, q4 = mape.direction_coeffs(p["qr"], p["qc"], p["qv"], p["w"], inst.n, G)
        mid = (p["l"] + p["u"]).float() / 2
        half = (p["u"] - p["l"]).float() / 4
        X0 = (mid + (torch.rand((case["S"], inst.n), generator=g, device=DEV) * 2 - 1) * half).round().to(torch.int32)
        return dict(kind=kind, n=inst.n, G=G, a=a, q4=q4, X0=X0, X=torch.empty_like(X0), iters=case["iters"], **p)
    if kind == "initial":
        inst = _instance(case["family"], case["n"], seed)
        l, u = _dev(inst.l), _dev(inst.u)
        X0 = l.float() + torch.rand((case["P"], inst.n), generator=g, device=DEV) * (u - l).float()
        lds = mape.round16(inst.n)
        z = torch.empty_like(X0)
        return dict(kind=kind, n=inst.n, A=_dev(inst.A), b=_dev(inst.b), l=l, u=u, X0=X0, X=z, M=torch.empty_like(z),
                    V=torch.empty_like(z), T=case["T"], lds=lds,
                    sol=torch.zeros((case["P"] * 16, lds), dtype=torch.uint8, device=DEV),
                    count=torch.zeros(1, dtype=torch.int64, device=DEV),
                    flags=torch.zeros(1, dtype=torch.int32, device=DEV),
                    kept=torch.zeros((case["P"] * 16, lds), dtype=torch.int8, device=DEV))
    if kind == "handle":
        inst = _instance(case["family"], case["n"], seed)
        cfg = mape.default_config(T=case["T"], precision=mape.PREC_BF16)
        rows = min(case["P"] * (case["T"] + 1), 1 << 18)
        return dict(kind=kind, inst=inst, cfg=cfg, P=case["P"], G0=I.uniform_samples(inst, case["P"], seed).G0,
                    kept=torch.zeros((rows, inst.n), dtype=torch.int8, pin_memory=True).numpy())
    insts = _uneven_instances(case, seed)
    cfg = mape.default_config(T=case["T"], precision=mape.PREC_BF16)
    server = mape.Server(cfg, max_slots=16)
    starts = [I.normal_starts(x, case["P"], case["std"], seed * 1000 + i).Z0 for i, x in enumerate(insts)]
    return dict(kind=kind, insts=insts, server=server, starts=starts, P=case["P"])


# ---------------------------------------------------------------------------
# one pass

def _begin(c):
    c["Z"].copy_(c["Z0"])
    c["M"].zero_()
    c["V"].zero_()
    c["cand_count"].zero_()
    c["flags"].zero_()


def _fill(dst, rows):
    dst[:rows.shape[0]].copy_(rows)
    return dst


def _union(c):
    k = min(int(c["cand_count"].item()), c["cand"].shape[0])
    rows = mape.dedup(c["cand"], k, c["n"])
    return _fill(c["kept"], rows), rows.shape[0]


def run(s):
    kind = s["kind"]
    if kind == "extract":
        c, cfg = s["call"], s["cfg"]
        _begin(c)
        mape.extract(c["B"], c["span"], c["Z"], c["M"], c["V"], t0=0, T=cfg.T, cfg=cfg, cand=c["cand"],
                     cand_count=c["cand_count"], flags=c["flags"], ldc=c["ldc"], workspace=c["workspace"])
        directions, K = _union(c)
        return dict(Z=c["Z"], M=c["M"], V=c["V"], flags=c["flags"], directions=directions, K=K)
    if kind == "batch":
        cfg = s["cfg"]
        keys = ("B", "span", "Z", "M", "V", "cand", "cand_count", "flags", "ldc", "workspace")
        for c in s["calls"]:
            _begin(c)
        mape.extract_batch([{k: c[k] for k in keys} for c in s["calls"]], t0=0, T=cfg.T, cfg=cfg)
        counts = torch.stack([c["cand_count"][0] for c in s["calls"]]).tolist()
        sets = mape.dedup_batch([(c["cand"], min(k, c["cand"].shape[0]), c["n"], None)
                                 for c, k in zip(s["calls"], counts)])
        # one tensor per kind of output: the instances' arrays one after the other
        cat = lambda k: torch.cat([c[k].reshape(-1) for c in s["calls"]])  # noqa: E731
        out = dict(Z=cat("Z"), M=cat("M"), V=cat("V"), K=torch.tensor([k for _, k, _ in sets]))
        for i, (c, (rows, _, _)) in enumerate(zip(s["calls"], sets)):
            out[f"directions{i}"] = _fill(c["kept"], rows)
        return out
    if kind == "project":
        return mape.project_starts(s["B"], s["G0"])
    if kind == "filter":
        n = s["n"]
        G = mape.dedup(s["cand"], s["cand"].shape[0], n)
        ok, fails = mape.kernel_test(s["A"], G, n)
        keep, rows = mape.minimal_filter(G, n, valid=ok)
        a, q4 = mape.direction_coeffs(s["qr"], s["qc"], s["qv"], s["w"], n, rows)
        return dict(ok=_fill(s["ok"], ok), keep=_fill(s["keep"], keep), rows=_fill(s["rows"], rows),
                    a=_fill(s["a"], a), q4=_fill(s["q4"], q4), fails=fails, K=G.shape[0])
    if kind == "augment":
        s["X"].copy_(s["X0"])
        fval, iters, moves, nmoves = mape.augment_run(s["G"], s["n"], s["a"], s["q4"], s["qr"], s["qc"], s["qv"], s["c"],
                                                  s["w"], s["l"], s["u"], s["X"], max_iters=s["iters"], moves_cap=s["iters"])
        return dict(X=s["X"], f=fval, iters=iters, moves=moves, nmoves=nmoves)
    if kind == "initial":
        s["X"].copy_(s["X0"])
        s["M"].zero_()
        s["V"].zero_()
        s["count"].zero_()
        mape.initial_solutions(s["A"], s["b"], s["l"], s["u"], s["X"], s["M"], s["V"], t0=0, T=s["T"], sol=s["sol"],
                               sol_count=s["count"], flags=s["flags"], lds=s["lds"])
        k = min(int(s["count"].item()), s["sol"].shape[0])
        points = mape.dedup(s["sol"].view(torch.int8), k, s["n"])
        return dict(X=s["X"], M=s["M"], V=s["V"], points=_fill(s["kept"], points), K=points.shape[0])
    if kind == "handle":
        inst = s["inst"]
        with mape.Instance.from_generated(inst, s["cfg"]) as h:
            h.extract_directions(s["P"], G0=s["G0"])
            h.wait()
            h.augment(inst.xbar[None, :])
            h.wait()
            x, f = h.solution()
            K = h.directions_i8(out=s["kept"]).shape[0]
            return dict(directions=s["kept"], K=K, x=x, f=f)
    server = s["server"]
    ids = [server.submit(x, s["P"], Z0=z) for x, z in zip(s["insts"], s["starts"])]
    server.wait_all()
    out = []
    for i in ids:
        out.append((*server.result(i), server.info(i)["directions"]))
        server.release(i)
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without

def _extract_work(n, m, P, T, period):
    """State and starts in, state out, B in; per start and step the products
    B' z and B'^T sign(B z) over the m rows below the identity, about 25
    operations per coordinate (gradient terms, Adam, rounding), and on the
    collecting steps B' round(z)."""
    d = n - m
    return dict(bytes=4.0 * P * d * 5 + 4.0 * n * d,
                flops=float(P) * T * (4.0 * m * d + 25.0 * d) + float(P) * (T // period) * 2.0 * m * d)


def _dims(case):
    n = case["n"]
    return n, max(1, n // (4 if case.get("family") == "small" else 5))


def work(case):
    kind = case["kind"]
    if kind == "extract":
        n, m = _dims(case)
        return _extract_work(n, m, case["P"], case["T"], case["period"])
    if kind in ("batch", "serve"):
        lo, hi, k = case["n_lo"], case["n_hi"], case["count"]
        tot = dict(bytes=0.0, flops=0.0)
        for i in range(k):
            n = int(round(lo * (hi / lo) ** (i / max(1, k - 1))))
            P = case["P"] * (4 if kind == "batch" and i % 3 == 2 else 1)
            w = _extract_work(n, max(1, n // 5), P, case["T"], 1)
            tot = dict(bytes=tot["bytes"] + w["bytes"], flops=tot["flops"] + w["flops"])
        return tot
    n, m = _dims(case)
    d = n - m
    if kind == "project":
        # the Gram matrix, its factor, the two triangular solves of W's n rows, the product with the samples
        return dict(bytes=4.0 * (case["P"] * (n + d) + n * d),
                    flops=float(n) * d * d + d ** 3 / 3.0 + 2.0 * n * d * d + 2.0 * case["P"] * n * d)
    if kind == "filter":
        # rows in, the distinct three quarters out, 17 bytes of flags and coefficients per row; A and Q per row
        K, ld = case["K"], mape.round16(n)
        nnz = m + 0.1 * m * d + 0.05 * n * n / 2
        return dict(bytes=K * ld * 1.75 + 17.0 * K, flops=2.0 * 0.75 * K * nnz)
    if kind == "augment":
        # at least one scoring pass over the set for every start
        K, ld = 0.75 * case["K"], mape.round16(n)
        return dict(bytes=K * ld + 16.0 * K, flops=2.0 * K * n * case["S"])
    if kind == "initial":
        return dict(bytes=4.0 * case["P"] * n * 4 + 4.0 * m * n,
                    flops=float(case["P"]) * case["T"] * (4.0 * m * n + 25.0 * n))
    w = _extract_work(n, m, case["P"], case["T"], 1)
    return dict(bytes=w["bytes"] + 4.0 * case["P"] * n, flops=w["flops"])


# ---------------------------------------------------------------------------
# the same in 64 bits

def _exact_extract(c, T, dt=torch.float64):
    """T Adam steps on Eq. (3) from the case's starts, in 64 bits."""
    l1, l2, lr, b1, b2, eps = 0.85, 1.0, 0.003, 0.9, 0.999, 1e-8
    # the weights and the step as the call's configuration holds them (FP32)
    l1, l2, lr, eps = (float(np.float32(v)) for v in (l1, l2, lr, eps))
    B = c["B"].to(dt)
    z = c["Z0"].to(dt)
    m, v = torch.zeros_like(z), torch.zeros_like(z)
    for t in range(1, T + 1):
        grad = torch.sign(z @ B.T) @ B + l1 * (z.ceil() + z.floor() - 2 * z)
        zi, k = z.abs().max(dim=1)
        on = (zi < 1) & (zi > 0)
        r = torch.arange(z.shape[0], device=z.device)
        grad[r, k] += torch.where(on, -l2 * torch.sign(z[r, k]) / (zi * zi), torch.zeros_like(zi))
        m = b1 * m + (1 - b1) * grad
        v = b2 * v + (1 - b2) * grad * grad
        z = z - lr * (m / (1 - b1 ** t)) / ((v / (1 - b2 ** t)).sqrt() + eps)
    return z, m, v


def _exact_project(s):
    B = s["B"].double()
    return torch.linalg.solve(B.T @ B, B.T @ s["G0"].double().T).T.contiguous()


def _exact_initial(s):
    lr, lam, b1, b2, eps = (float(np.float32(0.003)), float(np.float32(0.1)), 0.9, 0.999, float(np.float32(1e-8)))
    A, b, l, u = s["A"].double(), s["b"].double(), s["l"].double(), s["u"].double()
    x = torch.minimum(torch.maximum(s["X0"].double(), l), u)
    m, v = torch.zeros_like(x), torch.zeros_like(x)
    for t in range(1, s["T"] + 1):
        g = 2 * (x @ A.T - b) @ A + lam * (x.ceil() + x.floor() - 2 * x)
        m = b1 * m + (1 - b1) * g
        v = b2 * v + (1 - b2) * g * g
        x = x - lr * (m / (1 - b1 ** t)) / ((v / (1 - b2 ** t)).sqrt() + eps)
        x = torch.minimum(torch.maximum(x, l), u)
    return x, m, v


SIGNS_MOST = 60


def exact(case, seed):
    """The floating outputs in 64 bits.  Algorithm 2's steps depend on the
    signs of B z: a sign that 64 bits decide otherwise changes the gradient, and
    from there the two paths part.  The first moment, which follows the signs
    of the last steps, says something up to SIGNS_MOST steps, z and the second
    moment over a whole call, and nothing does where z enters B z with 4 or 8
    bits (e4m3, one BF16 term)."""
    kind = case["kind"]
    if kind == "extract":
        n, m = _dims(case)
        flops = 4.0 * case["P"] * n * (n - m) * case["T"]
        if case["prec"] != "bf16" or flops > 3e12:
            return None
        s = prepare(case, seed)
        z, mm, v = _exact_extract(s["call"], case["T"])
        return dict(Z=z, M=mm if case["T"] <= SIGNS_MOST else None, V=v, flags=None, directions=None, K=None)
    if kind == "batch":
        if work(case)["flops"] > 1e12:
            return None
        s = prepare(case, seed)
        parts = [_exact_extract(c, case["T"]) for c in s["calls"]]
        cat = lambda i: torch.cat([p[i].reshape(-1) for p in parts])  # noqa: E731
        return dict(Z=cat(0), M=cat(1), V=cat(2), K=None)
    if kind == "project":
        return _exact_project(prepare(case, seed))
    if kind == "initial":
        x, m, v = _exact_initial(prepare(case, seed))
        return dict(X=x, M=m, V=v, points=None, K=None)
    return None
