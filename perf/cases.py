"""Performance cases: what a user of the solver has it do, through the public binding
(``paper_2407_16144_gb300.rhpdhg``), over the range of linear programs the repository is built for.

Four kinds of pass:

* ``call``:  a new LP, start to finish: create (upload or device arrays, validation, transpose,
  scaling, step size), solve, poll, free.
* ``solve``: a kept handle is solved again and its solution polled into device memory; this is the
  iteration itself, which dominates every long solve.
* ``batch``: a kept batched solver takes a set of small LPs, advances them together and gives their
  results back.
* ``check``: the relative KKT error of a given point of an LP in device memory.

The LPs are the repository's own families (standard-form planted LPs, power-law general-form LPs,
multicommodity flow, planted infeasible LPs) at its own sizes and between them.  Iteration counts
are fixed through ``max_iters`` with a tolerance that is not met, except for ``infeasible``, which
runs until its certificate.  Every solve keeps the default restart, check and step settings.
Large LPs are drawn on the GPU, so that a preparation costs little; small ones come from
``lpgen``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2407_16144_gb300 import lpgen, rhpdhg

DEV = "cuda"


# ---- the cases ---------------------------------------------------------------------------------

def listed():
    return [
        # one small request, 200 x 500, plain rHPDHG in FP64 from host arrays: launches and the
        # fixed costs of a call are everything
        dict(name="call_200x500_fp64", kind="call", family="standard", m=200, n=500, alg=0, prec=0,
             host=True, iters=576),
        # a request of the serving stream above the batched size, mixed precision, host arrays
        dict(name="call_6kx15k_mixed", kind="call", family="standard", m=6000, n=15000, alg=1,
             prec=1, host=True, iters=640),
        # an infeasible LP in FP64, run to its certificate; sizes that are no multiple of a tile
        dict(name="call_infeasible_fp64", kind="call", family="infeasible", m=12_503, n=25_006,
             alg=1, prec=0, host=True, iters=20_000),
        # the headline LP (power-law columns, mixed bounds), the iteration in mixed precision
        dict(name="solve_c2_mixed", kind="solve", family="general", m=100_000, n=250_000, alg=1,
             prec=1, iters=512),
        # the same LP in FP64
        dict(name="solve_c2_fp64", kind="solve", family="general", m=100_000, n=250_000, alg=1,
             prec=0, iters=256),
        # the same LP new, from device arrays: set-up and the first iterations
        dict(name="call_c2_mixed", kind="call", family="general", m=100_000, n=250_000, alg=1,
             prec=1, host=False, iters=64),
        # multicommodity flow beyond the L2 cache: the iteration in the three precisions
        dict(name="solve_mcf_fp32", kind="solve", family="mcf", nodes=125_000, arcs=1_000_000,
             com=20, alg=1, prec=1, iters=96),
        dict(name="solve_mcf_bf16", kind="solve", family="mcf", nodes=62_500, arcs=500_000, com=20,
             alg=1, prec=2, iters=128),
        dict(name="solve_mcf_fp64", kind="solve", family="mcf", nodes=62_500, arcs=500_000, com=20,
             alg=0, prec=0, iters=96),
        # a new large LP: set-up is as long as many hundred iterations
        dict(name="call_mcf_bf16", kind="call", family="mcf", nodes=62_500, arcs=500_000, com=20,
             alg=1, prec=2, host=False, iters=64),
        # 96 small LPs advancing together as batched slots in mixed precision
        dict(name="batch_96_mixed", kind="batch", family="stream", count=96, m_lo=100, m_hi=1600,
             alg=1, prec=1, iters=256),
        # a solution checked against its LP
        dict(name="check_mcf", kind="check", family="mcf", nodes=62_500, arcs=500_000, com=20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["call_host", "call_host", "solve_general", "solve_general", "call_general",
                       "solve_mcf", "solve_mcf", "call_mcf", "batch", "check", "infeasible"])
    alg = rng.choice([0, 1, 1])
    if kind == "call_host":
        m = _log(rng, 100, 60_000)
        return dict(kind="call", family="standard", m=m, n=int(2.5 * m) + rng.randrange(7),
                    alg=alg, prec=rng.choice([0, 1]), host=True,
                    iters=64 * rng.randrange(2, 11))
    if kind in ("solve_general", "call_general"):
        m = _log(rng, 3000, 100_000)
        c = dict(kind=kind.split("_")[0], family="general", m=m, n=int(2.5 * m) + rng.randrange(7),
                 alg=alg, prec=rng.choice([0, 1]), iters=64 * rng.randrange(1, 5))
        if c["kind"] == "call":
            c["host"] = rng.random() < 0.5
        return c
    if kind in ("solve_mcf", "call_mcf"):
        nodes = _log(rng, 2000, 62_500)
        c = dict(kind=kind.split("_")[0], family="mcf", nodes=nodes,
                 arcs=8 * nodes + rng.randrange(9), com=rng.randrange(4, 21), alg=alg,
                 prec=rng.choice([0, 1, 2]), iters=64)
        if c["kind"] == "call":
            c["host"] = False
        return c
    if kind == "batch":
        return dict(kind="batch", family="stream", count=_log(rng, 1, 200), m_lo=100,
                    m_hi=_log(rng, 300, 1600), alg=alg, prec=rng.choice([0, 1]),
                    iters=64 * rng.randrange(1, 5))
    if kind == "infeasible":
        m = _log(rng, 500, 20_000)
        return dict(kind="call", family="infeasible", m=m, n=2 * m, alg=1, prec=0, host=True,
                    iters=20_000)
    if rng.random() < 0.5:
        m = _log(rng, 200, 100_000)
        return dict(kind="check", family="general", m=m, n=int(2.5 * m) + rng.randrange(7))
    nodes = _log(rng, 1000, 62_500)
    return dict(kind="check", family="mcf", nodes=nodes, arcs=8 * nodes + rng.randrange(9),
                com=rng.randrange(2, 21))


# ---- inputs ------------------------------------------------------------------------------------

def _sum_rows(ptr, v):
    return torch.segment_reduce(v, "sum", offsets=ptr, unsafe=True)


def _columns(row_ptr, col_idx, n):
    """Row indices, the order of the entries by column, and the column pointers of a CSR."""
    m = row_ptr.numel() - 1
    rows = torch.repeat_interleave(torch.arange(m, device=DEV), row_ptr[1:] - row_ptr[:-1])
    order = torch.argsort(col_idx, stable=True)
    cp = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    cp[1:] = torch.cumsum(torch.bincount(col_idx, minlength=n), 0)
    return rows, order, cp


def _general(seed, m, n):
    """A general-form LP in device memory: 70% equality rows, columns of power-law degree (exponent
    2.1, mean near 10, at most 5000), values +-1, integers to 10 and lognormal, half the variables
    in [0, inf), 30% boxed, 20% free, and a planted primal-dual optimum."""
    g = torch.Generator(device=DEV).manual_seed(seed)

    def uniform(k, lo=0.0, hi=1.0):
        return lo + (hi - lo) * torch.rand(k, generator=g, device=DEV, dtype=torch.float64)

    def normal(k):
        return torch.randn(k, generator=g, device=DEV, dtype=torch.float64)

    m_eq = (7 * m) // 10
    d = np.arange(2, min(5000, m // 4) + 1, dtype=np.float64)
    cdf = torch.from_numpy(np.cumsum(d ** -2.1) / np.sum(d ** -2.1)).to(DEV)
    deg = 2 + torch.searchsorted(cdf, uniform(n)).clamp_(max=len(d) - 1)
    cols = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    rows = torch.randint(0, m, (cols.numel(),), generator=g, device=DEV)
    key = torch.unique(rows * n + cols)
    rows, col = key // n, (key % n).to(torch.int32)
    nz = key.numel()
    row_ptr = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=m), 0)
    kind = uniform(nz)
    whole = torch.randint(1, 11, (nz,), generator=g, device=DEV).double()
    val = torch.where(kind < 0.3, 1.0, torch.where(kind < 0.6, whole, torch.exp(normal(nz))))
    val = torch.where(uniform(nz) < 0.5, -val, val)
    bound = uniform(n)
    low, box = bound < 0.5, (bound >= 0.5) & (bound < 0.8)
    lb = uniform(n, -10.0, 0.0)
    ub = lb + uniform(n, 1.0, 10.0)
    l = torch.where(low, 0.0, torch.where(box, lb, -math.inf))
    u = torch.where(box, ub, math.inf)
    pick, lam = uniform(n), uniform(n, 0.5, 2.0)
    x = torch.where(low, torch.where(pick < 0.4, 0.0, uniform(n, 0.5, 2.0)), normal(n))
    inner = lb + uniform(n) * (ub - lb)
    x = torch.where(box, torch.where(pick < 1 / 3, lb, torch.where(pick < 2 / 3, ub, inner)), x)
    lam = torch.where(low & (pick < 0.4), lam,
                      torch.where(box & (pick < 1 / 3), lam,
                                  torch.where(box & (pick < 2 / 3), -lam, 0.0)))
    y = normal(m)
    active = uniform(m - m_eq) < 0.5
    y[m_eq:] = torch.where(active, uniform(m - m_eq, 0.5, 2.0), 0.0)
    q = _sum_rows(row_ptr, val * x[col.long()])
    q[m_eq:] -= torch.where(active, 0.0, uniform(m - m_eq, 0.5, 2.0))
    _, order, cp = _columns(row_ptr, col, n)
    c = _sum_rows(cp, (val * y[rows])[order]) + lam
    return lpgen.LP(m_eq=m_eq, m_ineq=m - m_eq, n=n, row_ptr=row_ptr, col_idx=col, val=val, c=c,
                    q=q, l=l, u=u, x_star=x, y_star=y)


def _mcf(seed, nodes, arcs, com):
    """Multicommodity min-cost flow in device memory: a random cycle plus random arcs in
    forward-star order, flow conservation per commodity and node, one capacity row per arc, costs
    U[1, 100], capacities U[5, 50], supplies of a planted flow; every coefficient +-1."""
    g = torch.Generator(device=DEV).manual_seed(seed)

    def uniform(k, lo, hi):
        return lo + (hi - lo) * torch.rand(k, generator=g, device=DEV, dtype=torch.float64)

    perm = torch.randperm(nodes, generator=g, device=DEV)
    a = torch.randint(0, nodes, (arcs - nodes,), generator=g, device=DEV)
    b = torch.randint(0, nodes - 1, (arcs - nodes,), generator=g, device=DEV)
    key = torch.cat([perm * nodes + perm.roll(-1), a * nodes + b + (b >= a)]).sort().values
    tail, head = key // nodes, key % nodes
    arc = torch.arange(arcs, device=DEV)
    key, order = torch.cat([tail * arcs + arc, head * arcs + arc]).sort()
    sign = torch.where(order < arcs, 1.0, -1.0).double()
    ptr = torch.zeros(nodes + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.cumsum(torch.bincount(key // arcs, minlength=nodes), 0)
    k = torch.arange(com, device=DEV)
    conserve = (key % arcs)[None, :] + arcs * k[:, None]
    shared = arc[:, None] + arcs * k[None, :]
    col = torch.cat([conserve.reshape(-1).int(), shared.reshape(-1).int()])
    val = torch.cat([sign.repeat(com), torch.full((com * arcs,), -1.0, device=DEV).double()])
    rp = torch.cat([(ptr[None, :-1] + 2 * arcs * k[:, None]).reshape(-1),
                    2 * arcs * com + com * torch.arange(arcs + 1, device=DEV)])
    cost, cap = uniform(arcs, 1.0, 100.0), uniform(arcs, 5.0, 50.0)
    flow = uniform(com * arcs, 0.0, 1.0) * (cap / com).repeat(com)
    q = _sum_rows(rp[:com * nodes + 1], (val * flow[col.long()])[:2 * arcs * com])
    n = com * arcs
    return lpgen.LP(m_eq=com * nodes, m_ineq=arcs, n=n, row_ptr=rp, col_idx=col, val=val,
                    c=cost.repeat(com), q=torch.cat([q, -cap]),
                    l=torch.zeros(n, device=DEV).double(),
                    u=torch.full((n,), math.inf, device=DEV).double(), x_star=flow)


_ARRAYS = ("row_ptr", "col_idx", "val", "c", "q", "l", "u")


def _moved(lp, to_host):
    """The LP with its arrays in host memory (numpy) or in device memory (torch)."""
    out = lpgen.LP(lp.m_eq, lp.m_ineq, lp.n, *[getattr(lp, f) for f in _ARRAYS])
    for f in _ARRAYS:
        v = getattr(lp, f)
        if to_host and isinstance(v, torch.Tensor):
            setattr(out, f, v.cpu().numpy())
        elif not to_host and isinstance(v, np.ndarray):
            setattr(out, f, torch.from_numpy(v).to(DEV))
    return out


def _lp(case, seed):
    f = case["family"]
    if f == "standard":
        return lpgen.make_standard_planted(seed=seed, m=case["m"], n=case["n"])
    if f == "infeasible":
        return lpgen.make_primal_infeasible(seed, case["m"], case["n"])
    if f == "general":
        return _general(seed, case["m"], case["n"])
    return _mcf(seed, case["nodes"], case["arcs"], case["com"])


def _stream(case, seed):
    """Small requests of the serving stream: m spread over the logarithm of its range, arriving in
    no order of size, n = 2.5 m."""
    k = case["count"]
    at = (0.5 + (np.arange(k) * 0.6180339887498949) % 1.0 * (k - 1)) / k
    ms = case["m_lo"] * (case["m_hi"] / case["m_lo"]) ** at
    return [lpgen.make_standard_planted(seed=1000 + i + 7919 * (seed % 100_003), m=int(m),
                                        n=int(round(2.5 * int(m)))) for i, m in enumerate(ms)]


def _point(lp, seed):
    """A point near the planted flow or optimum, as a solve leaves it: x within the bounds."""
    g = torch.Generator(device=DEV).manual_seed(seed + 1)
    x = lp.x_star + 1e-3 * torch.randn(lp.n, generator=g, device=DEV, dtype=torch.float64)
    x = torch.minimum(torch.maximum(x, lp.l), lp.u)
    y = torch.randn(lp.m, generator=g, device=DEV, dtype=torch.float64)
    if lp.y_star is not None:
        y = lp.y_star + 1e-3 * y
    y[lp.m_eq:].clamp_(min=0.0)
    return x, y


def _params(case):
    return dict(algorithm=case["alg"], precision=case["prec"], eps_rel_kkt=1e-14,
                max_iters=case["iters"])


def prepare(case, seed):
    if case["kind"] == "batch":
        lps = _stream(case, seed)
        need = 0
        for lp in lps:
            keep = []
            need += rhpdhg.rhpdhg_batch_bytes_needed(rhpdhg.host_problem(lp, keep), case["prec"])
        return dict(case=case, lps=lps, batch=rhpdhg.Batch(case["count"], need + (1 << 20)))
    lp = _lp(case, seed)
    if case["kind"] == "check":
        x, y = _point(lp, seed)
        return dict(case=case, lp=lp, prob=rhpdhg.device_problem(lp), x=x, y=y)
    m, n = lp.m_eq + lp.m_ineq, lp.n
    st = dict(case=case, m=m, n=n)
    if case["kind"] == "solve":
        st["x"], st["y"] = (torch.empty(k, dtype=torch.float64, device=DEV) for k in (n, m))
        st["solver"] = rhpdhg.Solver(_moved(lp, False), device=True, **_params(case))
    else:
        st["lp"] = _moved(lp, case["host"])
    return st


# ---- passes ------------------------------------------------------------------------------------

def _numbers(r, prec):
    """What a solve gives back.  A mixed-precision point is handed on in FP32, the precision in
    which its iterates are held."""
    x, y = r.x, r.y
    if prec:
        if isinstance(x, np.ndarray):
            x, y = x.astype(np.float32), y.astype(np.float32)
        else:
            x, y = x.float(), y.float()
    return dict(x=x, y=y, objective=float(r.primal_obj), dual_objective=float(r.dual_obj),
                status=r.status, iters=r.iters, restarts=r.restarts)


def run(state):
    case = state["case"]
    if case["kind"] == "check":
        rc, out = rhpdhg.rhpdhg_kkt_eval(state["prob"], state["x"].data_ptr(),
                                         state["y"].data_ptr())
        assert rc == rhpdhg.OK
        return np.array(out)
    if case["kind"] == "solve":
        s = state["solver"]
        s.solve(1)
        return _numbers(s.poll(x=state["x"], y=state["y"], out_memory=rhpdhg.MEM_DEVICE),
                        case["prec"])
    if case["kind"] == "call":
        if case["host"]:
            with rhpdhg.Solver(state["lp"], **_params(case)) as s:
                r = s.run()
        else:
            x, y = (torch.empty(state[k], dtype=torch.float64, device=DEV) for k in ("n", "m"))
            with rhpdhg.Solver(state["lp"], device=True, **_params(case)) as s:
                s.solve(1)
                r = s.poll(x=x, y=y, out_memory=rhpdhg.MEM_DEVICE)
        out = _numbers(r, case["prec"])
        if case["family"] == "infeasible":
            out.update(cert_y=r.cert_y, source=r.cert_source)
        return out
    b = state["batch"]
    slots = [b.add(lp, **_params(case)) for lp in state["lps"]]
    res = b.run_all(slots, iters=64)
    got = [_numbers(res[s], case["prec"]) for s in slots]
    return {k: np.concatenate([np.atleast_1d(r[k]) for r in got]) for k in got[0]}


# ---- work ----------------------------------------------------------------------------------------

def _sizes(case):
    if case["family"] == "mcf":
        m = case["com"] * case["nodes"] + case["arcs"]
        n = case["com"] * case["arcs"]
        return m, n, 3 * n
    per = {"standard": 5, "general": 10, "infeasible": 6}[case["family"]]
    return case["m"], case["n"], per * case["n"]


def _iteration(m, n, nnz, prec, alg):
    """Bytes and flops of one iteration: both orientations of the matrix, the two gathered vectors
    and the vectors the updates read and write, each once."""
    v = {0: 8, 1: 4, 2: 2}[prec]
    w = 4 if prec else 8
    rows = (6 if prec else 7) + 4 * alg
    cols = (5 if prec else 7) + 4 * alg
    return (2 * nnz * (v + 4) + 4 * (m + n) + w * ((rows + 1) * m + (cols + 1) * n),
            4 * nnz + 23 * m + 19 * n)


def work(case):
    if case["kind"] == "batch":
        a, b = case["m_lo"], case["m_hi"]
        m = (b - a) / math.log(b / a)                # mean of the log-uniform sizes
        parts = [(m, 2.5 * m, 12.5 * m)] * case["count"]
    else:
        parts = [_sizes(case)]
    nbytes = flops = 0.0
    for m, n, nnz in parts:
        lp = 12 * nnz + 8 * (m + 1) + 8 * (3 * n + m)
        if case["kind"] == "check":
            nbytes += lp + 8 * (m + n)
            flops += 4 * nnz + 10 * (m + n)
            continue
        it, fl = _iteration(m, n, nnz, case["prec"], case["alg"])
        iters = 1400 if case["family"] == "infeasible" else case["iters"]
        nbytes += iters * it + 8 * (m + n)
        flops += iters * fl
        if case["kind"] != "solve":
            nbytes += lp
            # the power iteration: 201 products
            nbytes += 100.5 * (2 * nnz * ({0: 8, 1: 4, 2: 2}[case["prec"]] + 4) + 16 * (m + n))
            flops += 100.5 * 4 * nnz
    return dict(bytes=nbytes, flops=flops)


# ---- the results in 64 bits ----------------------------------------------------------------------

class _Matrix:
    """K and its transpose in torch's CSR, FP64, scaled as D K E once `scale` has run."""

    def __init__(self, lp):
        self.m, self.n = lp.m_eq + lp.m_ineq, lp.n
        self.rp, self.col, self.val = lp.row_ptr, lp.col_idx.long(), lp.val
        self.rows, self.order, self.cp = _columns(self.rp, self.col, self.n)
        self.D = torch.ones(self.m, dtype=torch.float64, device=DEV)
        self.E = torch.ones(self.n, dtype=torch.float64, device=DEV)

    def stat(self, how):
        a = (self.D[self.rows] * self.val * self.E[self.col]).abs()
        get = lambda k, i: torch.zeros(k, dtype=torch.float64, device=DEV).scatter_reduce_(  # noqa
            0, i, a, how)
        return get(self.m, self.rows), get(self.n, self.col)

    def scale(self, pow2):
        for how in ["amax"] * 10 + ["sum"]:
            r, c = self.stat(how)
            self.D = torch.where(r > 0, self.D / r.sqrt(), self.D)
            self.E = torch.where(c > 0, self.E / c.sqrt(), self.E)
        if pow2:
            for name in ("D", "E"):
                f, e = torch.frexp(getattr(self, name))
                setattr(self, name, torch.ldexp(torch.ones_like(f),
                                                e - (f < math.sqrt(0.5)).int()))
        v = self.D[self.rows] * self.val * self.E[self.col]
        self.K = torch.sparse_csr_tensor(self.rp, self.col, v, (self.m, self.n))
        self.KT = torch.sparse_csr_tensor(self.cp, self.rows[self.order], v[self.order],
                                          (self.n, self.m))

    def sigma(self):
        v = torch.full((self.n,), 1.0 / math.sqrt(self.n), dtype=torch.float64, device=DEV)
        for _ in range(100):
            v = self.KT @ (self.K @ v)
            v /= v.norm()
        return float((self.K @ v).norm())


def _solve64(lp, case):
    """Restarted Halpern PDHG (rHPDHG, or r2HPDHG for alg 1) with the library's default rules."""
    lp = _moved(lp, False)
    M = _Matrix(lp)
    M.scale(case["prec"] == 2)
    K, KT, D, E = M.K, M.KT, M.D, M.E
    c, q, l, u, m_eq = lp.c * E, lp.q * D, lp.l / E, lp.u / E, lp.m_eq
    eta = 0.9 / M.sigma()
    cn, qn = float(c.norm()), float(q.norm())
    omega = cn / qn if cn > 1e-10 and qn > 1e-10 else 1.0
    x = torch.minimum(torch.maximum(torch.zeros_like(c), l), u)
    y = torch.zeros_like(q)
    kx, ky = K @ x, KT @ y
    x0, y0, kx0, ky0 = x, y, kx, ky
    k = epoch = 0
    fpr0 = 0.0
    cert = None

    def farkas(d, kd):
        obj = float(q @ d)
        return obj > 0 and float((kd / E).clamp(min=0.0).max()) / obj <= 1e-8

    for t in range(case["iters"]):
        tau, sig = eta / omega, eta * omega
        xt = torch.minimum(torch.maximum(x - tau * (c - ky), l), u)
        kxt = K @ xt
        yt = y + sig * (q - 2.0 * kxt + kx)
        yt[m_eq:].clamp_(min=0.0)
        kyt = KT @ yt
        dx, dy = x - xt, y - yt
        fpr = float(dx @ dx) / tau + float(dy @ dy) / sig + 2.0 * float(dy @ (kx - kxt))
        if k == 0:
            fpr0 = fpr
        if case["family"] == "infeasible" and ((t + 1) % 64 == 0 or (k == 0 and epoch > 0)):
            if farkas(yt - y, kyt - ky):
                cert = D * (yt - y)
                break
        if t + 1 == case["iters"]:
            break
        if (epoch == 0 and k > 64) or (epoch > 0 and fpr <= math.exp(-2.0) * fpr0) or k >= 1000:
            if case["family"] == "infeasible" and farkas(yt - y0, kyt - ky0):
                cert = D * (yt - y0)
                break
            a, b = float((xt - x0).norm()), float((yt - y0).norm())
            if a > 1e-10 and b > 1e-10 and math.isfinite(b / a):
                omega = math.exp(0.5 * math.log(b / a) + 0.5 * math.log(omega))
            x, y, kx, ky = xt, yt, kxt, kyt
            x0, y0, kx0, ky0 = x, y, kx, ky
            k, epoch = 0, epoch + 1
            continue
        w = (k + 1.0) / (k + 2.0)
        r = 1.0 + case["alg"]
        x, y, kx, ky = (w * (r * v - (r - 1.0) * p) + (1.0 - w) * z for v, p, z in
                        ((xt, x, x0), (yt, y, y0), (kxt, kx, kx0), (kyt, ky, ky0)))
        k += 1
    lam = _reduced(c - kyt, l, u)
    pobj, dobj = float(c @ xt), float(q @ yt) + _bounds(lam, l, u)
    return dict(x=E * xt, y=D * yt, objective=pobj, dual_objective=dobj, cert_y=cert)


def _reduced(g, l, u):
    lf, uf = torch.isfinite(l), torch.isfinite(u)
    return torch.where(lf & uf, g, torch.where(lf, g.clamp(min=0.0),
                                               torch.where(uf, g.clamp(max=0.0), 0.0)))


def _bounds(lam, l, u):
    at = torch.where(lam > 0, l, torch.where(lam < 0, u, 0.0))
    return float((at * lam).sum())


def _kkt64(lp, x, y):
    M = _Matrix(lp)
    kx = torch.sparse_csr_tensor(M.rp, M.col, M.val, (M.m, M.n)) @ x
    ky = torch.sparse_csr_tensor(M.cp, M.rows[M.order], M.val[M.order], (M.n, M.m)) @ y
    r = lp.q - kx
    r[lp.m_eq:].clamp_(min=0.0)
    g = lp.c - ky
    lam = _reduced(g, lp.l, lp.u)
    p, d = float(lp.c @ x), float(lp.q @ y) + _bounds(lam, lp.l, lp.u)
    return np.array([float(r.norm()) / (1.0 + float(lp.q.norm())),
                     float((g - lam).norm()) / (1.0 + float(lp.c.norm())),
                     abs(p - d) / (1.0 + abs(p) + abs(d)), p, d])


def exact(case, seed):
    if case["kind"] == "check":
        lp = _lp(case, seed)
        return _kkt64(lp, *_point(lp, seed))
    if case["kind"] == "batch":
        if case["count"] * case["iters"] > 26_000:
            return None
        got = [_solve64(lp, case) for lp in _stream(case, seed)]
        return {k: (torch.cat([r[k] for r in got]) if k in ("x", "y")
                    else np.array([r[k] for r in got]))
                for k in ("x", "y", "objective", "dual_objective")}
    r = _solve64(_lp(case, seed), case)
    out = dict(x=r["x"], y=r["y"], objective=r["objective"], dual_objective=r["dual_objective"])
    if case["family"] == "infeasible":
        out = dict(cert_y=r["cert_y"])
    return out
