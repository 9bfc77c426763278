"""Performance cases: the work this framework is used for, through its public entry points.

A case is one of four calls a user's program makes:

* ``solve``: an LP that was created once is solved again from its initial point (``reset``, ``solve`` for a
  given number of step attempts, ``result``): the iteration that every solve spends its time in;
* ``create``: the whole call on host arrays: ``Problem(lp)`` (validation, copy, layout, preprocessing), a solve,
  the result, and the problem freed -- what a program with a new LP each time pays, and the serving loop's
  admission;
* ``batch``: one round of a batch of LPs in the batched kernel, from their initial points, and every result;
* ``norm``: the no-allocation power-norm estimate on a matrix that is already on the device.

The LPs are synthetic, made on the GPU from the seed: uniform random equality LPs, transportation LPs, LPs whose rows
have very different lengths ("linking" constraints among short ones), and LPs with power-law column degrees and
values over six decades.  A solve runs a fixed number of attempts (tolerance 0): the adaptive step makes the
iteration sensitive to rounding, so that after a few check periods two correct runs no longer agree, and
time-to-tolerance would count that and not the code's speed.  For the same reason a mixed-precision run with the
adaptive step is short, and ends in its FP32 phase, whose point is returned as the single-precision numbers it is.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2506_17650_gb300 as lpop

DEV = "cuda"
F64 = torch.float64


# ---------------------------------------------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------------------------------------------

def listed():
    def solve(name, family, m, n, nnz, mode, precision, alpha, attempts, check_every=64):
        return dict(name=name, call="solve", family=family, m=m, n=n, nnz=nnz, mode=mode, precision=precision,
                    alpha=alpha, attempts=attempts, check_every=check_every)

    return [
        # the smallest LP a program solves, vanilla step with the online update: all latency
        solve("tiny random, plain", "random", 200, 500, 2_500, "plain", "fp64", 1e-2, 256),
        # a small LP of the batch's size range solved by itself (a batch's tail, a served request)
        solve("small random", "random", 4_001, 10_003, 60_018, "pdlp", "fp64", 1e-3, 64),
        # ragged rows: a few rows of up to 3000 entries among short ones, odd sizes
        solve("linking rows", "linking", 1_003, 8_005, 376_000, "pdlp", "fp64", 1e-6, 64),
        # the medium transportation LP
        solve("transport", "transport", 50_000, 200_000, 400_000, "pdlp", "fp64", 1e-6, 64),
        # the same in mixed precision, with a check every 16 attempts
        solve("transport, mixed", "transport", 50_000, 200_000, 400_000, "pdlp", "mixed", 1e-6, 16, 16),
        # the middle of the serving stream's sizes
        solve("power law 1e6", "powerlaw", 66_667, 166_667, 1_000_000, "pdlp", "fp64", 1e-6, 64),
        # the large sparse LP, in both precisions
        solve("power law 3e7", "powerlaw", 2_000_000, 5_000_000, 30_000_000, "pdlp", "fp64", 1e-6, 64),
        solve("power law 3e7, mixed", "powerlaw", 2_000_000, 5_000_000, 30_000_000, "pdlp", "mixed", 1e-6, 16, 16),
        # a new LP of the serving stream: everything from host arrays to the result
        dict(solve("new power law 3e6", "powerlaw", 200_000, 500_000, 3_000_000, "pdlp", "fp64", 1e-6, 64),
             call="create"),
        # many small LPs in one launch, FP32 phase: 256 of them, as many sizes
        dict(name="batch, mixed", call="batch", family="random", members=256, m_lo=100, m_hi=20_000, cluster=1,
             wide_nnz=0, mode="plain", precision="mixed", alpha=1e-6, attempts=128, check_every=64),
        # fewer and larger ones, FP64, with clusters for the largest
        dict(name="batch, clusters", call="batch", family="random", members=64, m_lo=1_000, m_hi=20_000, cluster=4,
             wide_nnz=100_000, mode="pdlp", precision="fp64", alpha=1e-6, attempts=64, check_every=64),
        # ||A||_2 for a caller that owns all device memory
        dict(name="power norm", call="norm", family="random", m=120_000, n=300_000, nnz=1_800_000, iters=200),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["solve"] * 6 + ["create"] * 2 + ["batch"] * 2 + ["norm"])
    if call == "norm":
        m = _log(rng, 500, 150_000)
        n = int(m * rng.uniform(0.8, 2.5))
        return dict(call="norm", family="random", m=m, n=n, nnz=n * rng.randint(2, 8), iters=rng.choice([50, 100, 200]))
    precision = rng.choice(["fp64", "fp64", "mixed"])
    mode = rng.choice(["pdlp", "pdlp", "plain"])
    alpha = rng.choice([0.0, 1e-7, 1e-6, 1e-5, 1e-3])
    if call == "batch":
        if precision == "mixed":
            mode = "plain"
        lo = _log(rng, 60, 3_000)
        return dict(call="batch", family="random", members=rng.randint(16, 256), m_lo=lo,
                    m_hi=min(20_000, lo * rng.randint(2, 40)), cluster=rng.choice([1, 1, 2, 4, 8]),
                    wide_nnz=_log(rng, 20_000, 200_000), mode=mode, precision=precision, alpha=alpha,
                    attempts=rng.choice([48, 64]) if mode == "pdlp" else rng.choice([64, 128]), check_every=64)
    family = rng.choice(["random", "transport", "linking", "powerlaw", "powerlaw"])
    if family == "transport":
        n = _log(rng, 300, 1_000_000)
        m = max(20, int(n * rng.uniform(0.1, 0.5)))
        nnz = 2 * n
    elif family == "linking":
        n = _log(rng, 500, 60_000)
        m = max(30, int(n * rng.uniform(0.05, 0.5)))
        nnz = int(n * rng.uniform(6.0, 20.0))
        if precision == "mixed":
            mode = "plain"
    elif family == "powerlaw":
        nnz = _log(rng, 1_000, 12_000_000)
        n = nnz // 6
        m = max(10, int(n * rng.uniform(0.3, 0.5)))
    else:
        m = _log(rng, 60, 400_000)
        n = int(m * rng.uniform(1.5, 3.0))
        nnz = n * rng.randint(3, 8)
    if call == "create" and nnz > 6_000_000:
        nnz, n, m = nnz // 4, max(n // 4, 1), max(m // 4, 10)
    check_every = 64
    if mode == "plain":
        attempts = rng.choice([64, 100, 128, 192]) if nnz < 2_000_000 else 64
    elif precision == "mixed":
        attempts = check_every = 16
    else:
        attempts = rng.choice([64, 64, 64, rng.randint(33, 64)])  # sometimes a limit off a check
    return dict(call=call, family=family, m=m, n=n, nnz=nnz, mode=mode, precision=precision, alpha=alpha,
                attempts=attempts, check_every=check_every)


# ---------------------------------------------------------------------------------------------------------------
# Inputs (made on the GPU; every sum in a fixed order, so that a seed always gives the same bits)
# ---------------------------------------------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _rand(g, k):
    return torch.rand(k, generator=g, device=DEV, dtype=F64)


def _randn(g, k):
    return torch.randn(k, generator=g, device=DEV, dtype=F64)


def _offsets(idx, rows):
    """Row pointers of sorted row indices."""
    return torch.searchsorted(idx, torch.arange(rows + 1, device=DEV, dtype=idx.dtype))


def _rowsum(v, offsets):
    if v.numel() == 0:
        return torch.zeros(offsets.numel() - 1, device=DEV, dtype=v.dtype)
    return torch.segment_reduce(v, "sum", offsets=offsets, initial=0.0)


def _distinct(key):
    key, _ = torch.sort(key)
    keep = torch.ones_like(key, dtype=torch.bool)
    keep[1:] = key[1:] != key[:-1]
    return key[keep]


def _pattern(g, family, m, n, nnz):
    """Distinct entries (column * m + row, ascending)."""
    if family == "random":  # about nnz / n entries a column, uniform rows
        per = max(1, round(nnz / n))
        if n * per == nnz:
            deg = torch.full((n,), per, device=DEV, dtype=torch.int64)
        else:
            deg = torch.randint(max(1, per - 2), per + 3, (n,), generator=g, device=DEV)
    elif family == "powerlaw":  # column degrees with exponent 2.1, at most 1e5
        tail = _rand(g, n).clamp_(min=1e-15) ** (-1.0 / 1.1)
        dmax = min(100_000, m)
        lo, hi = 1e-6, float(nnz) / n
        for _ in range(60):
            mid = 0.5 * (lo + hi)
            if float(torch.clamp(torch.ceil(mid * tail), max=dmax).sum()) < nnz:
                lo = mid
            else:
                hi = mid
        deg = torch.clamp(torch.ceil(hi * tail), max=dmax).to(torch.int64)
    else:  # linking: row lengths log-uniform between 1 and min(n, 3000), scaled to nnz entries in all
        raw = torch.exp(_rand(g, m) * math.log(min(n, 3000)))
        deg = torch.clamp((raw * (nnz / float(raw.sum()))).round(), min=1, max=min(n, 3000)).to(torch.int64)
        rows = torch.repeat_interleave(torch.arange(m, device=DEV), deg)
        cols = torch.randint(0, n, (rows.numel(),), generator=g, device=DEV)
        return _distinct(cols * m + rows)
    cols = torch.repeat_interleave(torch.arange(n, device=DEV), deg)
    rows = torch.randint(0, m, (cols.numel(),), generator=g, device=DEV)
    return _distinct(cols * m + rows)


def _lp(family, m, n, nnz, seed):
    """An LP with the entries of A in CSR order, on the device."""
    g = _gen(seed)
    if family == "transport":
        S = max(1, m // 2)
        D = max(1, m - S)
        m = S + D
        k = torch.arange(n, device=DEV)
        src = torch.randint(0, S, (n,), generator=g, device=DEV)
        dst = torch.randint(0, D, (n,), generator=g, device=DEV)
        src[: min(S, n)] = k[: min(S, n)]  # every node has an arc
        d = min(D, max(0, n - S))
        dst[S: S + d] = k[:d]
        key = torch.stack([k * m + src, k * m + S + dst], dim=1).reshape(-1)
        vals = torch.ones(key.numel(), device=DEV, dtype=F64)
    else:
        key = _pattern(g, family, m, n, nnz)
        if family == "powerlaw":
            mag = 10.0 ** (6.0 * _rand(g, key.numel()) - 3.0)
            vals = torch.where(_rand(g, key.numel()) < 0.5, -mag, mag)
        else:
            vals = _randn(g, key.numel())
    cols, rows = key // m, key % m
    col_off = _offsets(cols, n)
    order = torch.argsort(rows * n + cols)
    ri, ci, v = rows[order], cols[order], vals[order]
    row_off = _offsets(ri, m)
    inf = float("inf")
    if family == "transport":
        x0 = 10.0 * _rand(g, n)
        b = _rowsum(x0[ci], row_off)
        b[:S] *= 1.2
        sense = torch.full((m,), ord("E"), device=DEV, dtype=torch.uint8)
        sense[:S] = ord("L")
        c = 1.0 + 99.0 * _rand(g, n)
        lb = torch.zeros(n, device=DEV, dtype=F64)
        ub = torch.full((n,), inf, device=DEV, dtype=F64)
    else:
        # an optimal pair (x0, y0) by complementary slackness
        p_free, p_ineq = {"random": (0.0, 0.0), "powerlaw": (0.2, 0.7), "linking": (0.1, 0.5)}[family]
        free = _rand(g, n) < p_free
        lb = torch.where(free, -inf, 0.0).to(F64)
        ub = torch.where(free, inf, 10.0).to(F64)
        u = _rand(g, n)
        low, high = ~free & (u < 0.4), ~free & (u > 0.9)
        x0 = torch.where(free, _randn(g, n), 10.0 * _rand(g, n))
        x0 = torch.where(low, 0.0, torch.where(high, 10.0, x0)).to(F64)
        ineq = _rand(g, m) < p_ineq
        tight = _rand(g, m) < 0.5
        y0 = _randn(g, m)
        y0 = torch.where(ineq, torch.where(tight, -y0.abs(), 0.0), y0).to(F64)
        b = _rowsum(v * x0[ci], row_off) + torch.where(ineq & ~tight, _rand(g, m), 0.0)
        sense = torch.where(ineq, ord("L"), ord("E")).to(torch.uint8)
        z = _rand(g, n)
        c = _rowsum(vals * y0[rows], col_off) + torch.where(low, z, torch.where(high, -z, 0.0))
    return SimpleNamespace(m=m, n=n, row_off=row_off, ci=ci, ri=ri, v=v, b=b, c=c, lb=lb, ub=ub, sense=sense)


def _host(d):
    """The arrays a user's program hands over."""
    return SimpleNamespace(m=d.m, n=d.n, row_ptr=d.row_off.cpu().numpy(), col_idx=d.ci.to(torch.int32).cpu().numpy(),
                           val=d.v.cpu().numpy(), b=d.b.cpu().numpy(), c=d.c.cpu().numpy(), lb=d.lb.cpu().numpy(),
                           ub=d.ub.cpu().numpy(), sense=d.sense.cpu().numpy())


def _member_sizes(case, seed):
    """Sizes m, n of a batch's members: the same number of each size for every seed, in another order."""
    k = case["members"]
    lo, hi = math.log(case["m_lo"]), math.log(case["m_hi"])
    ms = [int(math.exp(lo + (hi - lo) * (i + 0.5) / k)) for i in range(k)]
    return [(ms[i], int(2.5 * ms[i])) for i in np.random.RandomState(seed % (1 << 31)).permutation(k)]


def _member(seed, i, m, n):
    return _lp("random", m, n, 6 * n + 1, int(seed) * 1009 + i)


# ---------------------------------------------------------------------------------------------------------------
# The calls
# ---------------------------------------------------------------------------------------------------------------

def _options(case):
    return dict(mode=lpop.LP_MODE_PLAIN if case["mode"] == "plain" else lpop.LP_MODE_PDLP,
                precision=lpop.LP_PREC_MIXED if case["precision"] == "mixed" else lpop.LP_PREC_FP64,
                alpha=case["alpha"], phi=20, check_every=case["check_every"])


def prepare(case, seed):
    if case["call"] == "norm":
        d = _lp(case["family"], case["m"], case["n"], case["nnz"], seed)
        order = torch.argsort(d.ci * d.m + d.ri)
        arrays = [d.row_off.to(torch.int32), d.ci.to(torch.int32), d.v, _offsets(d.ci[order], d.n).to(torch.int32),
                  d.ri[order].to(torch.int32), d.v[order]]
        arrays = [a.contiguous() for a in arrays]
        return dict(case=case, m=d.m, n=d.n, arrays=arrays)
    if case["call"] == "batch":
        problems = []
        for i, (m, n) in enumerate(_member_sizes(case, seed)):
            problems.append(lpop.Problem(_host(_member(seed, i, m, n)), **_options(case)))
        batch = lpop.Batch(problems, case["cluster"], case["wide_nnz"] if case["cluster"] > 1 else 1 << 62)
        return dict(case=case, problems=problems, batch=batch)
    lp = _host(_lp(case["family"], case["m"], case["n"], case["nnz"], seed))
    if case["call"] == "create":
        return dict(case=case, lp=lp)
    return dict(case=case, problem=lpop.Problem(lp, **_options(case)))


def _outputs(case, x, y, stats):
    x, y = torch.from_numpy(x), torch.from_numpy(y)
    residuals = torch.tensor([[s["rel_pres"], s["rel_dres"], s["rel_gap"]] for s in stats], dtype=F64)
    objectives = torch.tensor([[s["pobj"], s["dobj"]] for s in stats], dtype=F64)
    counts = torch.tensor([[s["iterations"], s["accepted"], s["restarts"]] for s in stats])
    if case["precision"] == "mixed":  # the point of an FP32 phase: single-precision numbers
        x, y, residuals, objectives = (t.to(torch.float32) for t in (x, y, residuals, objectives))
    return dict(x=x, y=y, residuals=residuals, objectives=objectives, counts=counts)


def run(state):
    case = state["case"]
    if case["call"] == "norm":
        stream = torch.cuda.current_stream().cuda_stream
        return lpop.lp_power_norm_noalloc(state["m"], state["n"], *[a.data_ptr() for a in state["arrays"]],
                                          iters=case["iters"], stream=stream)
    if case["call"] == "batch":
        for p in state["problems"]:
            p.reset()
        state["batch"].round(0.0, case["attempts"], case["attempts"])
        res = [p.result() for p in state["problems"]]
        return _outputs(case, np.concatenate([r[0] for r in res]), np.concatenate([r[1] for r in res]),
                        [r[2] for r in res])
    if case["call"] == "create":
        with lpop.Problem(state["lp"], **_options(case)) as p:
            p.solve(0.0, case["attempts"])
            x, y, st = p.result()
        return _outputs(case, x, y, [st])
    p = state["problem"]
    p.reset()
    p.solve(0.0, case["attempts"])
    x, y, st = p.result()
    return _outputs(case, x, y, [st])


def _work(case, m, n, nnz):
    """One pass over an LP: per attempt both products (matrix once each), the vectors once; a check reads the same
    matrices and forms the residuals; the point out."""
    a, e = case["attempts"], 4.0 if case["precision"] == "mixed" else 8.0
    checks = 1 + max(1, a // case["check_every"])
    avg = 1 if case["mode"] == "pdlp" else 0
    attempt = 2 * nnz * (4 + e) + e * (n * (7 + 2 * avg) + 4 + m * (7 + 2 * avg)) + m
    check = (1 + avg) * nnz * (4 + e) + e * (5 * n + 5 * m)
    flops = a * (4.0 * nnz + 12 * n + 14 * m) + checks * ((4.0 + 2 * avg) * nnz + 12 * (n + m))
    return attempt * a + check * checks + 8.0 * (n + m), flops


def work(case):
    if case["call"] == "norm":
        nnz, m, n = case["nnz"], case["m"], case["n"]
        return {"bytes": case["iters"] * (24.0 * nnz + 16.0 * (m + n)), "flops": case["iters"] * (4.0 * nnz + 3.0 * n)}
    if case["call"] == "batch":
        each = [_work(case, m, n, 6 * n) for m, n in _member_sizes(case, 0)]
        return {"bytes": sum(b for b, _ in each), "flops": sum(f for _, f in each)}
    m, n, nnz = case["m"], case["n"], case["nnz"]
    b, f = _work(case, m, n, nnz)
    if case["call"] == "create":  # the LP in, ten rounds of row and column norms over the matrix, the layout out
        b += 12.0 * nnz + 8.0 * (m + 3 * n) + 12 * 12.0 * nnz + 24.0 * nnz
        f += 12 * 4.0 * nnz
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------------------------------------------
# The same in 64 bits with plain torch: the method as the paper states it
# ---------------------------------------------------------------------------------------------------------------

class _Exact:
    """Preprocessing and iteration of one LP in 64 bits."""

    def __init__(self, d, case):
        self.case, self.m, self.n = case, d.m, d.n
        self.pdlp = case["mode"] == "pdlp"
        to_col = torch.argsort(d.ci * d.m + d.ri)
        col_off = _offsets(d.ci[to_col], d.n)
        v = d.v.clone()
        dr, dc = torch.ones(d.m, device=DEV, dtype=F64), torch.ones(d.n, device=DEV, dtype=F64)

        def reduce(vals, how, power=1.0):
            a = vals.abs() ** power if power != 1.0 else vals.abs()
            r = torch.segment_reduce(a, how, offsets=d.row_off, initial=0.0)
            c = torch.segment_reduce(a[to_col], how, offsets=col_off, initial=0.0)
            return r, c

        def apply(r, c):
            nonlocal v, dr, dc
            fr = torch.where(r > 0, 1.0 / torch.sqrt(r), 1.0)
            fc = torch.where(c > 0, 1.0 / torch.sqrt(c), 1.0)
            v = (v * fr[d.ri]) * fc[d.ci]
            dr, dc = dr * fr, dc * fc

        for _ in range(10):
            apply(*reduce(v, "max"))
        if self.pdlp:
            apply(*reduce(v, "sum"))
        else:
            r, c = reduce(v, "sum", 2.0)
            apply(torch.sqrt(r), torch.sqrt(c))
        self.A = torch.sparse_csr_tensor(d.row_off, d.ci, v, size=(d.m, d.n))
        self.At = torch.sparse_csr_tensor(col_off, d.ri[to_col], v[to_col], size=(d.n, d.m))
        self.dr, self.dc = dr, dc
        self.b, self.c = dr * d.b, dc * d.c
        self.l, self.u = d.lb / dc, d.ub / dc
        self.lf, self.uf = torch.isfinite(self.l), torch.isfinite(self.u)
        self.le, self.eq = d.sense == ord("L"), d.sense == ord("E")
        self.bn, self.cn = float(d.b.norm()), float(d.c.norm())
        bs, cs = float(self.b.norm()), float(self.c.norm())
        self.omega = cs / bs if bs > 0 and cs > 0 else 1.0
        self.eta = 1.0 / float(v.abs().max()) if self.pdlp else 0.9 / _power_norm(self.A, self.At, d.n, 200)
        self.x = torch.zeros(d.n, device=DEV, dtype=F64).clamp(self.l, self.u)
        self.y = torch.zeros(d.m, device=DEV, dtype=F64)
        self.ax = self.A @ self.x
        self.T, self.S = torch.ones_like(self.x), torch.ones_like(self.y)
        self.GT, self.GS = torch.zeros_like(self.x), torch.zeros_like(self.y)
        self.k = self.t = self.restarts = self.t_last = 0
        self.clear()
        self.x_last = None

    def clear(self):
        self.xbar, self.ybar, self.wsum = torch.zeros_like(self.x), torch.zeros_like(self.y), 0.0

    def attempt(self):
        eta, w, x, y, ax = self.eta, self.omega, self.x, self.y, self.ax
        g = self.c - self.At @ y
        xh = x - (eta / w) * self.T * g
        x1 = xh.clamp(self.l, self.u)
        ax1 = self.A @ x1
        r = self.b - (2.0 * ax1 - ax)
        yh = y + (eta * w) * self.S * r
        out = self.le & (yh > 0)
        y1 = torch.where(out, 0.0, yh)
        self.t += 1
        accept = True
        if self.pdlp:
            dx, dy = x1 - x, y1 - y
            move = w * float((dx * dx / self.T).sum()) + float((dy * dy / self.S).sum()) / w
            inter = abs(float((dy * (ax1 - ax)).sum()))
            limit = move / (2.0 * inter) if inter else math.inf
            accept = eta <= limit
            self.eta = min((1.0 - (self.t + 1) ** -0.3) * limit, (1.0 + (self.t + 1) ** -0.6) * eta)
        if not accept:
            return
        if self.k % 20 == 0:
            res = self.b - ax
            for P, G, grad, norm in (("T", "GT", (eta / w) * torch.where((xh >= self.l) & (xh <= self.u), g * g, 0.0), g),
                                     ("S", "GS", (eta * w) * torch.where(out, 0.0, res * r), res)):
                n2 = float((norm * norm).sum())
                if n2 <= 0:
                    continue
                grad = -grad / n2
                acc = getattr(self, G) + grad * grad
                step = torch.where(acc > 0, grad / torch.sqrt(acc), 0.0)
                setattr(self, G, acc)
                setattr(self, P, (getattr(self, P) - self.case["alpha"] * step).clamp(min=1e-6))
        if self.pdlp:
            self.xbar, self.ybar, self.wsum = self.xbar + eta * x1, self.ybar + eta * y1, self.wsum + eta
        self.x, self.y, self.ax = x1, y1, ax1
        self.k += 1

    def kkt(self, x, y, ax):
        rs = ax - self.b
        ps = torch.where(self.eq, rs, rs.clamp(min=0.0))
        rc = self.c - self.At @ y
        lam = torch.where(self.lf & self.uf, rc, torch.where(self.lf, rc.clamp(min=0.0),
                                                             torch.where(self.uf, rc.clamp(max=0.0), 0.0)))
        ds = rc - lam
        pobj = float(self.c @ x)
        dobj = float(self.b @ y) + float((torch.where(self.lf, self.l, 0.0) * lam.clamp(min=0.0)).sum()) \
            - float((torch.where(self.uf, self.u, 0.0) * (-lam).clamp(min=0.0)).sum())
        gap = pobj - dobj
        st = dict(pobj=pobj, dobj=dobj, rel_pres=float((ps / self.dr).norm()) / (1.0 + self.bn),
                  rel_dres=float((ds / self.dc).norm()) / (1.0 + self.cn),
                  rel_gap=abs(gap) / (1.0 + abs(pobj) + abs(dobj)))
        return st, (float(ps @ ps), float(ds @ ds), gap * gap)

    def weighted(self, p, w):
        return math.sqrt(w * w * p[0] + p[1] / (w * w) + p[2])

    def check(self):
        self.stats, parts = self.kkt(self.x, self.y, self.ax)
        if not self.pdlp:
            return
        if self.x_last is None:
            self.x_last, self.y_last, self.parts = self.x, self.y, parts
            self.k_prev = self.weighted(parts, self.omega)
            return
        cand = [(self.x, self.y, self.ax, parts)]
        if self.wsum > 0:
            xa, ya = self.xbar / self.wsum, self.ybar / self.wsum
            axa = self.A @ xa
            cand.append((xa, ya, axa, self.kkt(xa, ya, axa)[1]))
        ks = [self.weighted(c[3], self.omega) for c in cand]
        i = 1 if len(ks) > 1 and ks[1] < ks[0] else 0
        last = self.weighted(self.parts, self.omega)
        go = ks[i] <= 0.2 * last or (ks[i] <= 0.8 * last and ks[i] > self.k_prev) or self.t - self.t_last >= 0.36 * self.t
        self.k_prev = ks[i]
        if not go:
            return
        x, y, ax, parts = cand[i]
        dx, dy = float((x - self.x_last).norm()), float((y - self.y_last).norm())
        if dx > 1e-10 and dy > 1e-10:
            self.omega = math.exp(0.5 * math.log(dy / dx) + 0.5 * math.log(self.omega))
        self.x, self.y, self.ax, self.x_last, self.y_last, self.parts = x, y, ax, x, y, parts
        self.clear()
        self.t_last, self.restarts = self.t, self.restarts + 1

    def solve(self):
        self.check()
        every, limit = self.case["check_every"], self.case["attempts"]
        while self.t < limit:
            self.attempt()
            if self.t % every == 0:
                self.check()
        if self.t % every:
            self.stats = self.kkt(self.x, self.y, self.ax)[0]
        st = dict(self.stats, iterations=self.t, accepted=self.k, restarts=self.restarts)
        return (self.dc * self.x).cpu().numpy(), (self.dr * self.y).cpu().numpy(), st


def _power_norm(A, At, n, iters):
    v = torch.full((n,), 1.0 / math.sqrt(n), device=DEV, dtype=F64)
    nw = 0.0
    for _ in range(iters):
        w = At @ (A @ v)
        nw = w.norm()
        v = w / nw
    return math.sqrt(float(nw))


def exact(case, seed):
    if case["call"] == "norm":
        d = _lp(case["family"], case["m"], case["n"], case["nnz"], seed)
        to_col = torch.argsort(d.ci * d.m + d.ri)
        A = torch.sparse_csr_tensor(d.row_off, d.ci, d.v, size=(d.m, d.n))
        At = torch.sparse_csr_tensor(_offsets(d.ci[to_col], d.n), d.ri[to_col], d.v[to_col], size=(d.n, d.m))
        return _power_norm(A, At, d.n, case["iters"])
    if case["call"] == "batch":
        lps = [_member(seed, i, m, n) for i, (m, n) in enumerate(_member_sizes(case, seed))]
    else:
        lps = [_lp(case["family"], case["m"], case["n"], case["nnz"], seed)]
    res = [_Exact(d, case).solve() for d in lps]
    out = _outputs(dict(case, precision="fp64"), np.concatenate([r[0] for r in res]),
                   np.concatenate([r[1] for r in res]), [r[2] for r in res])
    return dict(out, counts=None)
