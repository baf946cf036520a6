"""The calls that a user of the LP solver makes, as measurable cases.

A case is one call (or one create / solve / destroy sequence) of the public
interface on an LP that is drawn on the GPU from a seed: the termination check
of a point, a restarted-PDHG or Halpern solve, a new LP solved from scratch, a
batch of LPs, the gradient of unrolled iterations and the multi-start cast.

Solves run a fixed number of iterations (their tolerance is out of reach), so a
pass is the same work for every seed; the row lengths of an LP depend on its size
alone, its columns and values on the seed.  The adaptive steps of Algorithm 5, the
library's default, amplify rounding tenfold every 15 to 30 iterations: they are
taken in FP64 and over one check period.  Longer solves and those with FP32
iterations take the fixed step; the launches are the same ones.  What an FP32
solve or an FP32 gradient returns is kept as FP32, as a program that works in that
precision keeps it.

``exact`` restates the published algorithms in 64 bits with torch alone.
"""
import math

import numpy as np
import torch

from paper_2508_16806_gb300 import autograd as A
from paper_2508_16806_gb300 import lp as L
from paper_2508_16806_gb300 import synth

PREC = {"fp64": L.LP_PREC_FP64, "mixed": L.LP_PREC_MIXED}
CHECK = 64            # accepted iterations between two KKT checks (the library's default)
GRAD_CKPT = 50        # iterations between two checkpoints of an unrolled run
TINY_TOL = 1e-30      # a tolerance that no solve reaches


def listed():
    return [
        # a serving process that checks a candidate point before it accepts it
        dict(name="kkt check 5k", do="kkt", shape="random", m=5000, prec="fp64"),
        # the 200 x 400 LP of the smoke test: latency, launches and control flow
        dict(name="solve 200x400 fp64", do="solve", shape="dense", m=200, prec="fp64", iters=256,
             method="fixed"),
        # one of the uneven LPs of the batch workload, solved by itself
        dict(name="solve 5k mixed", do="solve", shape="random", m=5000, prec="mixed", iters=512,
             method="fixed"),
        # the largest of those LPs in plain FP64
        dict(name="solve 50k fp64", do="solve", shape="random", m=50000, prec="fp64", iters=256,
             method="fixed"),
        # the Halpern variant on the LP of the gradient workload
        dict(name="halpern 100k mixed", do="solve", shape="random", m=100000, prec="mixed",
             iters=256, method="halpern"),
        # an LP that was not seen before, with the default options: copy, transpose, scaling,
        # schedules, solve, release
        dict(name="new lp 20k fp64", do="new", shape="random", m=20000, prec="fp64", iters=64,
             method="adaptive"),
        # the large power-law LP (about 20M nonzeros), FP32 iterations
        dict(name="solve 1M powerlaw mixed", do="solve", shape="powerlaw", m=1000000, prec="mixed",
             iters=256, method="fixed"),
        # the same in plain FP64 with adaptive steps
        dict(name="solve 1M powerlaw fp64", do="solve", shape="powerlaw", m=1000000, prec="fp64",
             iters=64, method="adaptive"),
        # the dispatch-shaped LP: 615,001 rows over 5,000 generators, about 38M nonzeros
        dict(name="dispatch 615k mixed", do="solve", shape="dispatch", m=15000, prec="mixed",
             iters=256, method="fixed"),
        # uneven LPs solved together, the batched form
        dict(name="batch of 64 mixed", do="batch", shape="random", m=50000, prec="mixed",
             iters=128, method="fixed", count=64),
        # gradient of 500 unrolled iterations, the differentiable form, in its default precision
        # (in FP32 a mask of the projections flips with the last bit: such runs are drawn short)
        dict(name="grad 100k fp64", do="grad", shape="random", m=100000, prec="fp64", iters=500),
        # multi-start warm start: 32 points, 20 steps a round
        dict(name="fishnet 50k mixed", do="fishnet", shape="random", m=50000, prec="mixed",
             points=32, iters=20),
    ]


def _log_int(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    do = rng.choice(["kkt", "solve", "solve", "solve", "large", "dispatch", "new", "batch", "grad",
                     "fishnet"])
    prec = rng.choice(["fp64", "mixed"])
    method = rng.choice(["fixed"] if prec == "mixed" else ["fixed", "adaptive"])

    def iters(lo, hi):
        return rng.randint(32, 64) if method == "adaptive" else rng.randint(lo, hi)

    if do == "kkt":
        return dict(do=do, shape="random", m=_log_int(rng, 200, 50000), prec="fp64")
    if do == "solve":
        m = _log_int(rng, 100, 100000)
        return dict(do=do, shape="dense" if m < 400 else rng.choice(["random", "powerlaw"]), m=m,
                    prec=prec, iters=iters(100, 300), method=rng.choice([method, method, "halpern"]))
    if do == "large":
        return dict(do="solve", shape="powerlaw", m=_log_int(rng, 200000, 1000000), prec=prec,
                    iters=iters(64, 128), method=rng.choice([method, method, "halpern"]))
    if do == "dispatch":
        return dict(do="solve", shape=do, m=_log_int(rng, 500, 15000), prec=prec,
                    iters=iters(64, 128), method=method)
    if do == "new":
        return dict(do=do, shape="random", m=_log_int(rng, 200, 50000), prec=prec,
                    iters=iters(32, 64), method=method)
    if do == "batch":
        return dict(do=do, shape="random", m=_log_int(rng, 2000, 50000), prec=prec,
                    iters=iters(64, 128), method=method, count=rng.randint(5, 32))
    if do == "grad":
        if prec == "fp64":
            return dict(do=do, shape="random", m=_log_int(rng, 50, 50000), prec=prec,
                        iters=rng.randint(20, 200))
        return dict(do=do, shape="random", m=_log_int(rng, 50, 2000), prec=prec,
                    iters=rng.randint(10, 30))
    return dict(do=do, shape="random", m=_log_int(rng, 500, 50000), prec=prec,
                points=2 ** rng.randint(2, 6), iters=rng.randint(5, 20))


# ----------------------------------------------------------------- the LPs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float64)


def _row_ptr(rows, m):
    rp = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(rows, minlength=m), 0)
    return rp


def _segment_sum(rows, v, count):
    """Sums of v by row, in an order of their own (no atomics: the same inputs every time)."""
    order = torch.argsort(rows, stable=True)
    return torch.segment_reduce(v[order], "sum", offsets=_row_ptr(rows, count), initial=0.0)


def _pattern(g, m, n, lengths):
    """lengths[i] distinct uniformly random columns in row i: (rows, cols), sorted."""
    rows = torch.repeat_interleave(torch.arange(m, device="cuda"), lengths)
    key = torch.sort(rows * n + torch.randint(0, n, rows.shape, generator=g, device="cuda"))[0]
    while True:
        again = torch.nonzero(key[1:] == key[:-1])[:, 0] + 1
        if not again.numel():
            return key // n, key % n
        key[again] = key[again] // n * n + torch.randint(0, n, again.shape, generator=g,
                                                         device="cuda")
        key = torch.sort(key)[0]


def _dispatch(g, m):
    """The dispatch-shaped LP: one balance row, m base flow rows with 10..200 shift factors over
    m / 3 generators, and 40 contingency blocks that repeat them with coefficients +-10 %."""
    n = max(m // 3, 500)
    pmin = 50.0 * _rand(g, n)
    pmax = pmin + 10.0 + 190.0 * _rand(g, n)
    x0 = pmin + (pmax - pmin) * _rand(g, n)
    lengths = torch.exp(math.log(10.0) + math.log(20.0) * _rand(_gen(m), m)).long()
    rows, cols = _pattern(g, m, n, lengths)
    base = 0.3 * _randn(g, rows.numel())
    blocks = [base] + [base * (0.9 + 0.2 * _rand(g, rows.numel())) for _ in range(40)]
    flow = torch.cat(blocks)
    r = torch.cat([rows + k * m for k in range(41)])
    ax0 = _segment_sum(r, flow * x0[cols].repeat(41), 41 * m)
    limit = ax0 + _rand(g, 41 * m) * ax0.abs() + 0.1
    rows = torch.cat([torch.zeros(n, dtype=torch.int64, device="cuda"), r + 1])
    cols = torch.cat([torch.arange(n, device="cuda"), cols.repeat(41)])
    sense = torch.ones(41 * m + 1, dtype=torch.uint8, device="cuda")
    sense[0] = 0
    return dict(m=41 * m + 1, n=n, rows=rows, cols=cols,
                vals=torch.cat([torch.ones(n, dtype=torch.float64, device="cuda"), -flow]),
                sense=sense, c=10.0 + 90.0 * _rand(g, n), q=torch.cat([x0.sum()[None], -limit]),
                l=pmin, u=pmax)


def _tensors(shape, m, seed):
    """One LP as CUDA tensors: rows and cols of the nonzeros, vals, sense, c, q, l, u."""
    g = _gen(seed)
    if shape == "dispatch":
        return _dispatch(g, m)
    n, fixed = 2 * m, _gen(m)
    if shape == "dense":            # 2 % of the entries
        lengths = (_rand(fixed, m, n) < 0.02).sum(1)
    elif shape == "powerlaw":       # P(length) ~ length^-2.1 on 4..5000
        pmf = torch.arange(4, 5001, device="cuda", dtype=torch.float64) ** -2.1
        cdf = torch.cumsum(pmf, 0) / pmf.sum()
        lengths = (4 + torch.searchsorted(cdf, _rand(fixed, m))).clamp(max=min(5000, n // 4))
    else:                           # 5 to 20 nonzeros in a row
        lengths = torch.randint(5, 21, (m,), generator=fixed, device="cuda")
    rows, cols = _pattern(g, m, n, lengths)
    vals = _randn(g, rows.numel())
    # a planted optimum (x0, y0): half >= rows, half = rows; 30 % of x0 at its lower bound and
    # 20 % at its upper one, with reduced costs of the matching sign
    sense = torch.zeros(m, dtype=torch.uint8, device="cuda")
    sense[: m - m // 2] = 1
    l, u = torch.zeros(n, dtype=torch.float64, device="cuda"), 1.0 + 4.0 * _rand(g, n)
    which = _rand(g, n)
    low, up = which < 0.3, (which >= 0.3) & (which < 0.5)
    x0 = torch.where(low, l, torch.where(up, u, _rand(g, n)))
    y0 = _randn(g, m)
    y0 = torch.where(sense.bool(), y0.clamp(min=0.0), y0)
    slack = torch.where(sense.bool() & (y0 == 0.0), _rand(g, m), 0.0)
    lam = torch.where(low, _rand(g, n), torch.where(up, -_rand(g, n), 0.0))
    return dict(m=m, n=n, rows=rows, cols=cols, vals=vals, sense=sense,
                c=_segment_sum(cols, vals * y0[rows], n) + lam,
                q=_segment_sum(rows, vals * x0[cols], m) - slack, l=l, u=u)


def _host_lp(t):
    def arr(v, dtype):
        return np.ascontiguousarray(v.cpu().numpy().astype(dtype, copy=False))

    return synth.LP(t["m"], t["n"], arr(_row_ptr(t["rows"], t["m"]), np.int64),
                    arr(t["cols"], np.int32), arr(t["vals"], np.float64),
                    arr(t["sense"], np.uint8), arr(t["c"], np.float64), arr(t["q"], np.float64),
                    arr(t["l"], np.float64), arr(t["u"], np.float64))


def _batch_sizes(case):
    """Rows of the LPs of a batch: log-uniform between a hundredth of m and m."""
    rng = np.random.default_rng(case["count"])
    return [max(int(case["m"] * math.exp(-v)), 20)
            for v in rng.uniform(0.0, math.log(100.0), case["count"])]


def _batch_lps(case, seed):
    return [_tensors(case["shape"], m, seed + 1000 * (k + 1))
            for k, m in enumerate(_batch_sizes(case))]


def _options(case):
    o = dict(precision=PREC[case["prec"]], tol=TINY_TOL, max_iters=case["iters"],
             check_every=CHECK)
    if case["prec"] == "mixed":
        o["polish_switch_tol"] = TINY_TOL
    if case["method"] == "fixed":
        o["adaptive_step"] = 0
    if case["method"] == "halpern":
        o["halpern"] = 1
    return o


# --------------------------------------------------------- prepare and run

class _State:
    """What the program holds: the LP's handle, its inputs, the stream they live on."""

    def __init__(self, case):
        self.case = case
        self.stream = torch.cuda.Stream()
        self.problem = self.batch = None


def prepare(case, seed):
    s = _State(case)
    do = case["do"]
    with torch.cuda.stream(s.stream):
        if do == "batch":
            s.batch = L.Batch([_host_lp(t) for t in _batch_lps(case, seed)])
            return s
        t = _tensors(case["shape"], case["m"], seed)
        g = _gen(seed + 1)
        s.lp = _host_lp(t)
        if do == "new":
            return s
        s.problem = L.Problem(s.lp, stream=s.stream)
        if do == "kkt":
            s.x = t["l"] + (t["u"] - t["l"]) * _rand(g, t["n"])
            s.y = _randn(g, t["m"])
        elif do == "grad":
            f = torch.float64 if case["prec"] == "fp64" else torch.float32
            s.leaves = [t[k].to(f).requires_grad_() for k in ("c", "q", "vals")]
            s.target = _rand(g, t["n"])
        elif do == "fishnet":
            s.G = _randn(g, t["n"], case["points"]).cpu().numpy()
            s.Z = np.random.default_rng(seed).standard_normal(
                max(L.lp_fishnet_draws(case["points"]), 1))
    s.stream.synchronize()
    return s


def _keep(case, *tensors):
    """Results of FP32 iterations as FP32."""
    if case["prec"] == "fp64":
        return list(tensors)
    return [v.to(torch.float32) if isinstance(v, torch.Tensor) else v.astype(np.float32)
            for v in tensors]


def _solved(case, problem):
    x, y, info, _ = problem.solve(out_device=True, **_options(case))
    return _keep(case, x, y) + [info["iters"], info["restarts"], info["status"]]


def run(s):
    case = s.case
    do = case["do"]
    with torch.cuda.stream(s.stream):
        if do == "kkt":
            return np.array(L.lp_kkt_noalloc(s.problem.desc, s.x.data_ptr(), s.y.data_ptr(), 1.5,
                                             s.stream.cuda_stream))
        if do == "solve":
            return _solved(case, s.problem)
        if do == "new":
            problem = L.Problem(s.lp, stream=s.stream)
            out = _solved(case, problem)
            problem.close()
            return out
        if do == "batch":
            res = s.batch.solve(**_options(case))
            x, y = _keep(case, np.concatenate([r[0] for r in res]),
                         np.concatenate([r[1] for r in res]))
            return [x, y, np.array([r[2]["iters"] for r in res]),
                    np.array([r[2]["restarts"] for r in res])]
        if do == "grad":
            x = A.UnrolledPDHG.apply(*s.leaves, s.problem, case["iters"], GRAD_CKPT,
                                     PREC[case["prec"]])
            loss = ((x - s.target) ** 2).sum()
            return _keep(case, x.detach()) + list(torch.autograd.grad(loss, s.leaves))
        x, y, gaps, rounds = s.problem.fishnet(case["points"], case["iters"], s.G, s.Z,
                                               precision=PREC[case["prec"]])
        return _keep(case, x, y, np.nan_to_num(gaps)) + [rounds]


# --------------------------------------------------------------- the work

def _nnz(case, m):
    """Expected nonzeros of an LP with m rows (of a block of base rows for dispatch)."""
    if case["shape"] == "dispatch":
        return 41 * m * (190.0 / math.log(20.0))
    if case["shape"] == "dense":
        return 0.04 * m * m
    return m * (20.0 if case["shape"] == "powerlaw" else 12.5)


def work(case):
    """Bytes and operations of one pass: the nonzeros (value and column index) and the vectors
    that each product with K or K^T takes, at the precision of the iterations; a pass over the
    FP64 input for what builds a new LP.  An iteration is two products, each on its own vector."""
    m, do = case["m"], case["do"]
    s = 8 if case["prec"] == "fp64" else 4
    if do == "batch":
        # the mean of exp(-U[0, ln 100])
        nnz, rows = (case["count"] * 0.99 / math.log(100.0) * v for v in (_nnz(case, m), m))
        cols = 2 * rows
    else:
        nnz, rows = _nnz(case, m), 41 * m if case["shape"] == "dispatch" else m
        cols = max(m // 3, 500) if case["shape"] == "dispatch" else 2 * m
    pair = 2 * nnz * (s + 4) + 4 * (rows + cols) * s
    if do == "kkt":
        return dict(bytes=12 * nnz + 8 * (3 * rows + 4 * cols), flops=4 * nnz)
    if do == "grad":
        # forward and reverse, and the derivative of every nonzero in FP64
        k = case["iters"]
        return dict(bytes=2 * k * pair + 8 * nnz, flops=k * (8 * nnz + 6 * nnz))
    if do == "fishnet":
        # the points of the rounds, each taking `iters` iterations
        p, cols_of, i = case["points"], [], 0
        while p > 1:
            cols_of.append(p)
            p = 2 * (p // 2) if i % 2 == 1 and p > 2 else p // 2
            i += 1
        k, pts = case["iters"], sum(cols_of)
        return dict(bytes=k * (len(cols_of) * 2 * nnz * (s + 4) + 4 * pts * (rows + cols) * s),
                    flops=4.0 * k * pts * nnz)
    more = 2 * 12 * nnz if do == "new" else 0
    return dict(bytes=case["iters"] * pair + more, flops=case["iters"] * 4.0 * nnz)


# -------------------------------------------------------------- 64 bits

class _Ref:
    """The scaled problem (Algorithm 3), its norm (Algorithm 2) and its products, in 64 bits."""

    def __init__(self, t, ruiz):
        self.m, self.n, rows, cols = t["m"], t["n"], t["rows"], t["cols"]
        v = t["vals"].clone()
        self.R = torch.ones(self.m, dtype=torch.float64, device="cuda")
        self.C = torch.ones(self.n, dtype=torch.float64, device="cuda")
        for _ in range(ruiz):
            a = v.abs()
            rn = torch.zeros_like(self.R).scatter_reduce_(0, rows, a, "amax")
            cn = torch.zeros_like(self.C).scatter_reduce_(0, cols, a, "amax")
            both = torch.cat([rn, cn])
            if (1.0 - both[both > 0]).abs().max() <= 1e-4:
                break
            r = torch.where(rn > 0, 1.0 / rn.sqrt(), 1.0)
            k = torch.where(cn > 0, 1.0 / cn.sqrt(), 1.0)
            v *= r[rows] * k[cols]
            self.R *= r
            self.C *= k
        self.K = torch.sparse_csr_tensor(_row_ptr(rows, self.m), cols, v, (self.m, self.n))
        order = torch.argsort(cols, stable=True)
        self.KT = torch.sparse_csr_tensor(_row_ptr(cols, self.n), rows[order], v[order],
                                          (self.n, self.m))
        self.c, self.q = self.C * t["c"], self.R * t["q"]
        self.l, self.u = t["l"] / self.C, t["u"] / self.C
        self.ge = t["sense"].bool()
        self.c0, self.q0 = t["c"], t["q"]
        b = torch.ones(self.n, dtype=torch.float64, device="cuda")
        for _ in range(100):
            b = self.KT @ (self.K @ b)
            b /= b.norm()
        self.norm = float((self.K @ b).norm())
        self.eta = 0.9 / self.norm
        self.omega = float(self.c.norm() / self.q.norm())

    def box(self, x):
        return torch.minimum(torch.maximum(x, self.l), self.u)

    def cone(self, y):
        return torch.where(self.ge, y.clamp(min=0.0), y)

    def start(self):
        x = self.box(torch.zeros(self.n, dtype=torch.float64, device="cuda"))
        return x, torch.zeros(self.m, dtype=torch.float64, device="cuda")

    def lam(self, y, kty):
        v = self.c - kty
        lf, uf = torch.isfinite(self.l), torch.isfinite(self.u)
        pos = torch.where(lf, v.clamp(min=0.0), 0.0)
        neg = torch.where(uf, v.clamp(max=0.0), 0.0)
        bound = torch.where(pos > 0, self.l * pos, 0.0).sum() + \
            torch.where(neg < 0, self.u * neg, 0.0).sum()
        return v - pos - neg, bound

    def kkt(self, x, y, kx, kty, w):
        r = self.q - kx
        r = torch.where(self.ge, r.clamp(min=0.0), r)
        d, bound = self.lam(y, kty)
        gap = self.q @ y + bound - self.c @ x
        return float((w * w * (r @ r) + (d @ d) / (w * w) + gap * gap).sqrt())


def _ref_solve(t, case):
    """Algorithm 1 with the restarts of Section 2.4.2, Algorithms 4 and 5, or Halpern steps."""
    P = _Ref(t, 10)
    halp, adaptive = case["method"] == "halpern", case["method"] == "adaptive"
    rho = (1.0 if case["prec"] == "fp64" else 0.5) if halp else 0.0
    eta, w = P.eta, P.omega
    x, y = P.start()
    kx, kty = P.K @ x, P.KT @ y
    xa, ya, kxa = x, y, kx                  # the anchor of the epoch
    xs, ys, W = torch.zeros_like(x), torch.zeros_like(y), 0.0
    k = epoch = restarts = 0
    anchor = P.kkt(x, y, kx, kty, w)
    prev = fpr_prev = math.inf
    fpr = fpr0 = 0.0
    cand = (x, y)
    while k < case["iters"]:
        tau, sigma = eta / w, eta * w
        xh = P.box(x - tau * (P.c - kty))
        kxh = P.K @ xh
        yh = P.cone(y + sigma * (P.q - (2.0 * kxh - kx)))
        dx, dy = xh - x, yh - y
        step, accept = eta, True
        if adaptive or halp:
            move = float(w * (dx @ dx) + (dy @ dy) / w)
            inter = float(dy @ (kxh - kx))
        if adaptive:
            bar = move / (2.0 * abs(inter)) if inter else math.inf
            accept = eta <= bar
            eta = min((1.0 - (k + 2.0) ** -0.3) * bar, (1.0 + (k + 2.0) ** -0.6) * eta)
        if not accept:
            continue
        if halp:
            fpr = math.sqrt(max(move / eta + 2.0 * inter, 0.0))
            fpr0 = fpr if epoch == 0 else fpr0
            lam = (epoch + 1.0) / (epoch + 2.0)
            a, b, g = lam * (1.0 + rho), lam * rho, 1.0 - lam
            x, y, kx = (a * xh - b * x + g * xa, a * yh - b * y + g * ya,
                        a * kxh - b * kx + g * kxa)
        else:
            x, y, kx = xh, yh, kxh
            xs, ys, W = xs + step * x, ys + step * y, W + step
        kty = P.KT @ y
        k, epoch = k + 1, epoch + 1
        if k % CHECK and k < case["iters"]:
            continue
        if halp:
            ax, ay, avg = xh, yh, True
        else:
            ax, ay = P.box(xs / W), P.cone(ys / W)
        kax, kay = P.K @ ax, P.KT @ ay
        now, mean = P.kkt(x, y, kx, kty, w), P.kkt(ax, ay, kax, kay, w)
        if not halp:
            avg = not now < mean
        err = mean if avg else now
        cand = (ax, ay) if avg else (x, y)
        if halp:
            again = fpr <= 0.2 * fpr0 or (fpr <= 0.8 * fpr0 and fpr > fpr_prev)
        else:
            again = err <= 0.2 * anchor or (err <= 0.8 * anchor and err > prev)
        if not (again or epoch > 0.36 * k):
            prev, fpr_prev = err, fpr
            continue
        ddx, ddy = float((cand[0] - xa).norm()), float((cand[1] - ya).norm())
        if ddx > 1e-6 and ddy > 1e-6:
            w = math.exp(0.5 * math.log(ddy / ddx) + 0.5 * math.log(w))
        if avg:
            x, y, kx, kty = ax, ay, kax, kay
        xa, ya, kxa = x, y, kx
        xs, ys, W = torch.zeros_like(x), torch.zeros_like(y), 0.0
        anchor, prev, fpr_prev, epoch, restarts = err, math.inf, math.inf, 0, restarts + 1
    return P.C * cand[0], P.R * cand[1], k, restarts


def _ref_grad(t, case, target):
    """Unrolled fixed steps on the unscaled problem and their reverse."""
    P = _Ref(t, 0)
    w = float(P.c.norm() / P.q.norm())
    tau, sigma = P.eta / w, P.eta * w
    x, y = P.start()
    kx, kty = P.K @ x, P.KT @ y
    xs, ys, mx, my = [x], [y], [], []
    for _ in range(case["iters"]):
        v = x - tau * (P.c - kty)
        x = P.box(v)
        kx1 = P.K @ x
        z = y + sigma * (P.q - (2.0 * kx1 - kx))
        y, kx = P.cone(z), kx1
        kty = P.KT @ y
        mx.append((P.l < v) & (v < P.u))
        my.append(~P.ge | (z > 0))
        xs.append(x)
        ys.append(y)
    gx, gy = 2.0 * (x - target), torch.zeros_like(y)
    dc, dq, dv = torch.zeros_like(x), torch.zeros_like(y), torch.zeros_like(t["vals"])
    rows, cols = t["rows"], t["cols"]
    for k in range(case["iters"] - 1, -1, -1):
        gvy = torch.where(my[k], gy, 0.0)
        dq += sigma * gvy
        gb = -sigma * (P.KT @ gvy)
        gvx = torch.where(mx[k], gx + 2.0 * gb, 0.0)
        dc -= tau * gvx
        dv += -sigma * gvy[rows] * (2.0 * xs[k + 1] - xs[k])[cols] + tau * ys[k][rows] * gvx[cols]
        gx, gy = gvx - gb, gvy + tau * (P.K @ gvx)
    return x, dc, dq, dv


def _ref_fishnet(t, case, G, Z):
    """Algorithm 7: cast, advance, cull by duality gap, repopulate."""
    P = _Ref(t, 10)
    tau, sigma = P.eta / P.omega, P.eta * P.omega
    X = (P.norm / math.sqrt(P.n)) * G
    Y = P.K @ X
    KX = Y.clone()
    gaps = np.zeros((18, case["points"]))
    rounds = pos = 0
    c, l, u, q, ge = (v[:, None] for v in (P.c, P.l, P.u, P.q, P.ge))
    while X.shape[1] > 1:
        top = X.shape[1]
        for _ in range(case["iters"]):
            X = torch.minimum(torch.maximum(X - tau * (c - P.KT @ Y), l), u)
            K1 = P.K @ X
            Y = Y + sigma * (q - (2.0 * K1 - KX))
            Y, KX = torch.where(ge, Y.clamp(min=0.0), Y), K1
        KTY = P.KT @ Y
        gap = torch.stack([(P.q @ Y[:, p] + P.lam(Y[:, p], KTY[:, p])[1] - P.c @ X[:, p]).abs()
                           for p in range(top)]).cpu().numpy()
        gaps[rounds, :top] = gap
        keep = top // 2
        kept = torch.from_numpy(np.sort(np.argsort(gap, kind="stable")[:keep])).cuda()
        X, Y, KX = X[:, kept], Y[:, kept], KX[:, kept]
        if rounds % 2 == 1 and top > 2:
            wts = np.abs(Z[pos:pos + keep * keep]).reshape(keep, keep)
            wts = torch.from_numpy(wts / wts.sum(1, keepdims=True)).cuda().T
            pos += keep * keep
            X, Y, KX = (torch.cat([V, V @ wts], 1) for V in (X, Y, KX))
        X, Y, KX = X.contiguous(), Y.contiguous(), KX.contiguous()
        rounds += 1
    return P.C * X[:, 0], P.R * Y[:, 0], gaps[:rounds], rounds


def exact(case, seed):
    do = case["do"]
    if do == "batch":
        res = [_ref_solve(t, case) for t in _batch_lps(case, seed)]
        return [torch.cat([r[0] for r in res]), torch.cat([r[1] for r in res]),
                np.array([r[2] for r in res]), np.array([r[3] for r in res])]
    t = _tensors(case["shape"], case["m"], seed)
    g = _gen(seed + 1)
    if do == "kkt":
        x, y = t["l"] + (t["u"] - t["l"]) * _rand(g, t["n"]), _randn(g, t["m"])
        r = t["q"] - _segment_sum(t["rows"], t["vals"] * x[t["cols"]], t["m"])
        r = torch.where(t["sense"].bool(), r.clamp(min=0.0), r)
        v = t["c"] - _segment_sum(t["cols"], t["vals"] * y[t["rows"]], t["n"])
        bound = (t["l"] * v.clamp(min=0.0) + t["u"] * v.clamp(max=0.0)).sum()
        pobj, dobj = float(t["c"] @ x), float(t["q"] @ y + bound)
        pres, gap = float(r.norm()), dobj - pobj      # finite bounds: no dual residual
        return np.array([pobj, dobj, pres, 0.0, abs(gap) / (1.0 + abs(dobj) + abs(pobj)),
                         pres / (1.0 + float(t["q"].norm())), 0.0,
                         math.sqrt(1.5 ** 2 * pres ** 2 + gap ** 2)])
    if do == "grad":
        f = torch.float64 if case["prec"] == "fp64" else torch.float32
        for k in ("c", "q", "vals"):
            t[k] = t[k].to(f).to(torch.float64)
        return list(_ref_grad(t, case, _rand(g, t["n"])))
    if do == "fishnet":
        G = _randn(g, t["n"], case["points"])
        Z = np.random.default_rng(seed).standard_normal(
            max(L.lp_fishnet_draws(case["points"]), 1))
        return list(_ref_fishnet(t, case, G, Z))
    x, y, iters, restarts = _ref_solve(t, case)
    return [x, y, iters, restarts, L.LP_ITERATION_LIMIT]
