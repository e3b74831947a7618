"""Timed cases: the work a user has the solver library do, through its public entry points.

A case is a dict of plain values; ``kind`` names the path:

  lp         one LP or QP solved for a bounded number of PDHG iterations
             (``pdlp.Solver.solve``): host arrays of x and y come back
  transport  one transportation LP solved from a warm start
  batch      many uneven LPs in one launch (``pdlp.BatchSolver.solve``)
  tbatch     many transportation LPs of one family from warm starts
  train      Adam steps of the warm-start network (``pdlp.Mlp.train``), the
             losses and the updated weights
  predict    the network's predictions on the host (``pdlp.Mlp.predict``)
  scale      the allocation-free scaling of a device-resident K and K'

Inputs are made on the GPU from the seed.  ``exact`` recomputes a case's
outputs in 64 bits with plain torch, without the library.  A solve stops
after a bounded number of iterations (a check period and a restart for one
LP, less for a batch): PDHG with adaptive steps amplifies rounding by orders
of magnitude in every further period, so that longer runs of two correct
programs can no longer be compared elementwise.
"""

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2311_12180_gb300 import pdlp as P

F64 = torch.float64


def listed():
    return [
        # the smallest LP a user solves: a few hundred rows, bound by latency
        dict(name="lp_tiny", kind="lp", pattern="uniform", m=200, n=500, nnz=2000, iters=80, tol=1e-8, bits=64, qp=False),
        # power-law LPs of the size sweep: 1e5 and 1e6 nonzeros
        dict(name="lp_1e5", kind="lp", pattern="zipf", m=5000, n=10000, nnz=100_000, iters=80, tol=1e-8, bits=64, qp=False),
        dict(name="lp_1e6", kind="lp", pattern="zipf", m=50_000, n=100_000, nnz=1_000_000, iters=80, tol=1e-8, bits=64, qp=False),
        # the headline LP, its FP32-values mode, and the same with a diagonal quadratic objective
        dict(name="lp_2e7", kind="lp", pattern="zipf", m=1_000_000, n=2_000_000, nnz=20_000_000, iters=80, tol=1e-8, bits=64, qp=False),
        dict(name="lp_2e7_f32", kind="lp", pattern="zipf", m=1_000_000, n=2_000_000, nnz=20_000_000, iters=80, tol=1e-8, bits=32, qp=False),
        dict(name="qp_2e7", kind="lp", pattern="zipf", m=1_000_000, n=2_000_000, nnz=20_000_000, iters=80, tol=1e-8, bits=64, qp=True),
        # one member of the 200 x 300 transportation family from a predicted start
        dict(name="transport_warm", kind="transport", sources=200, sinks=300, iters=40, tol=1e-8),
        # uneven LPs of the batch recipe (m log-uniform in 50..4000) in one launch
        dict(name="batch_uneven", kind="batch", count=256, m_lo=50, m_hi=4000, shapes=1, iters=48, tol=1e-9),
        # warm-started members of the transportation family in one launch
        dict(name="batch_transport", kind="tbatch", count=48, sources=200, sinks=300, iters=32, tol=1e-8),
        # the warm-start network of the 200 x 300 family: training and prediction
        dict(name="mlp_train", kind="train", hidden=256, out=60_500, batch=256, steps=64),
        dict(name="mlp_predict", kind="predict", hidden=256, out=60_500, count=500, max_batch=256),
        # scaling of a matrix that is already on the device, near the entry point's size limit
        dict(name="scale_3e6", kind="scale", m=150_000, n=250_000, nnz=3_000_000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["lp", "lp", "lp", "transport", "batch", "tbatch", "train", "predict", "scale"])
    if kind == "lp":
        nnz = _log(rng, 2000, 16_000_000)
        m = max(20, int(nnz / rng.uniform(12, 30)))
        n = max(30, int(m * rng.uniform(1.2, 2.4)))
        form = rng.choice(["lp", "lp", "f32", "qp"])
        pattern = "uniform" if nnz < 50_000 and rng.random() < 0.5 else "zipf"
        return dict(kind=kind, pattern=pattern, m=m, n=n, nnz=nnz, iters=rng.randrange(48, 81), tol=1e-8,
                    bits=32 if form == "f32" else 64, qp=form == "qp")
    if kind == "transport":
        return dict(kind=kind, sources=_log(rng, 8, 400), sinks=_log(rng, 12, 500), iters=rng.randrange(24, 41), tol=1e-8)
    if kind == "batch":
        lo = _log(rng, 30, 200)
        return dict(kind=kind, count=_log(rng, 12, 220), m_lo=lo, m_hi=_log(rng, 4 * lo, 4000), shapes=rng.randrange(1 << 20),
                    iters=rng.randrange(32, 49), tol=1e-9)
    if kind == "tbatch":
        s = _log(rng, 10, 200)
        k = int(s * rng.uniform(1.0, 1.5))
        return dict(kind=kind, count=_log(rng, 8, 46) if s > 60 else _log(rng, 20, 300), sources=s, sinks=k,
                    iters=rng.randrange(20, 33), tol=1e-8)
    if kind == "train":
        return dict(kind=kind, hidden=rng.choice([32, 64, 100, 128, 256]), out=_log(rng, 200, 60_000),
                    batch=rng.randrange(17, 257), steps=rng.randrange(16, 64))
    if kind == "predict":
        return dict(kind=kind, hidden=rng.choice([32, 64, 100, 128, 256]), out=_log(rng, 200, 60_000),
                    count=_log(rng, 1, 490), max_batch=256)
    nnz = _log(rng, 3000, 2_900_000)
    m = max(50, int(nnz / rng.uniform(12, 30)))
    return dict(kind=kind, m=min(m, 260_000), n=min(int(m * rng.uniform(0.8, 2.4)), 260_000), nnz=nnz)


# ---------------------------------------------------------------- inputs


def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1000003 + salt)
    return g


def _uni(g, size, lo=0.0, hi=1.0):
    return torch.rand(size, dtype=F64, device="cuda", generator=g) * (hi - lo) + lo


def _row_sums(a, lengths):
    """Sums of consecutive groups of a, in a fixed order."""
    return torch.segment_reduce(a, "sum", lengths=lengths, unsafe=True, initial=0.0)


def _zipf_lengths(g, m, n, nnz, alpha=1.5, cap=5000):
    """Power-law row lengths max(1, round(s Z)), Z ~ Zipf(alpha) clipped at
    `cap`, s chosen for `nnz` in total."""
    pmf = np.arange(1, cap + 1, dtype=np.float64) ** -alpha
    cdf = np.cumsum(pmf)
    cdf /= cdf[-1] + sum(k ** -alpha for k in range(cap + 1, 400_000, 7)) * 7
    z = torch.bucketize(_uni(g, m), torch.tensor(cdf, device="cuda")).clamp_(max=cap - 1) + 1
    hist = torch.bincount(z, minlength=cap + 1).cpu().numpy()
    ks = np.arange(cap + 1)
    lo, hi = 0.0, 1.0
    while (np.minimum(np.maximum(1, np.rint(hi * ks)), n) * hist).sum() < nnz and hi < 1e6:
        hi *= 2
    for _ in range(60):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if (np.minimum(np.maximum(1, np.rint(mid * ks)), n) * hist).sum() < nnz else (lo, mid)
    return (z.double() * hi).round().clamp_(min=1, max=n).long()


def _blocks(ms, ns, n_eqs):
    """Index maps of LPs laid side by side (block diagonal)."""
    t = lambda a: torch.tensor(np.asarray(a, dtype=np.int64), device="cuda")  # noqa: E731
    B = SimpleNamespace(count=len(ms), ms=t(ms), ns=t(ns), n_eqs=t(n_eqs))
    B.M, B.N = int(sum(ms)), int(sum(ns))
    ids = torch.arange(B.count, device="cuda")
    B.row_blk, B.col_blk = torch.repeat_interleave(ids, B.ms), torch.repeat_interleave(ids, B.ns)
    B.ro, B.co = t(np.concatenate([[0], np.cumsum(ms)])), t(np.concatenate([[0], np.cumsum(ns)]))
    B.ineq = (torch.arange(B.M, device="cuda") - B.ro[B.row_blk]) >= B.n_eqs[B.row_blk]
    return B


def _entries(g, B, lengths, cover):
    """Distinct uniform columns of each row (global row and column of every
    entry, row-major); with `cover` every column gets an entry."""
    rows = torch.repeat_interleave(torch.arange(B.M, device="cuda"), lengths)
    width = B.ns[B.row_blk[rows]]
    cols = B.co[B.row_blk[rows]] + (_uni(g, rows.numel()) * width).long().minimum(width - 1)
    if cover:
        empty = torch.nonzero(torch.bincount(cols, minlength=B.N) == 0).flatten()
        blk = B.col_blk[empty]
        r = B.ro[blk] + (_uni(g, empty.numel()) * B.ms[blk]).long().minimum(B.ms[blk] - 1)
        rows, cols = torch.cat([rows, r]), torch.cat([cols, empty])
    key = torch.unique(rows * B.N + cols)  # sorted
    return key // B.N, key % B.N


def _plant(g, B, rows, cols, val, l, u):
    """q and c of a planted optimal pair, as every generator of this
    repository plants one: 30 % of the bounded variables on a bound, half of
    the ">=" rows active."""
    N, M = B.N, B.M
    lf, uf = torch.isfinite(l), torch.isfinite(u)
    lo, hi = torch.where(lf, l, torch.zeros_like(l)), torch.where(uf, u, torch.zeros_like(u))
    r5 = _uni(g, N, 0.0, 5.0)
    x = torch.randn(N, dtype=F64, device="cuda", generator=g)
    x = torch.where(lf & uf, lo + (hi - lo) * _uni(g, N), torch.where(lf, lo + r5, torch.where(uf, hi - r5, x)))
    at = (_uni(g, N) < 0.3) & (lf | uf)
    low = at & lf & (~uf | (_uni(g, N) < 0.5))
    upp = at & uf & ~low
    x = torch.where(low, lo, torch.where(upp, hi, x))
    lam = _uni(g, N, 0.1, 1.0)
    lam = torch.where(low, lam, torch.where(upp, -lam, torch.zeros_like(lam)))
    y = torch.randn(M, dtype=F64, device="cuda", generator=g)
    active = _uni(g, M) < 0.5
    y = torch.where(B.ineq, torch.where(active, _uni(g, M, 0.1, 1.0), torch.zeros_like(y)), y)
    q = _row_sums(val * x[cols], torch.bincount(rows, minlength=M))
    q = torch.where(B.ineq & ~active, q - _uni(g, M, 0.1, 1.0), q)
    order = torch.argsort(cols, stable=True)
    c = _row_sums((val * y[rows])[order], torch.bincount(cols, minlength=N)) + lam
    return c, q, x


def _finish(B, rows, cols, val, c, q, l, u):
    ptr = torch.zeros(B.M + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(torch.bincount(rows, minlength=B.M), 0, out=ptr[1:])
    return SimpleNamespace(B=B, rows=rows, cols=cols, val=val, ptr=ptr, c=c, q=q, l=l, u=u, qd=None, x0=None, y0=None)


def _pattern(g, case, B):
    if case.get("pattern") == "uniform":
        dens = torch.full((case["m"],), case["nnz"] / (case["m"] * case["n"]), dtype=F64, device="cuda")
        lengths = torch.binomial(torch.full_like(dens, float(case["n"])), dens, generator=g).long().clamp_(min=1)
        return _entries(g, B, lengths, True)
    return _entries(g, B, _zipf_lengths(g, case["m"], case["n"], case["nnz"]), False)


def _lp(case, seed):
    """A planted LP: uniform sparsity with N(0, 1) values and 0 <= x <= 10, or
    power-law rows with lognormal values and mixed bounds."""
    g = _gen(seed, 1)
    m, n = case["m"], case["n"]
    B = _blocks([m], [n], [m // 2 if case["pattern"] == "uniform" else round(0.4 * m)])
    rows, cols = _pattern(g, case, B)
    val = torch.randn(rows.numel(), dtype=F64, device="cuda", generator=g)
    if case["pattern"] == "uniform":
        l, u = torch.zeros(n, dtype=F64, device="cuda"), torch.full((n,), 10.0, dtype=F64, device="cuda")
    else:
        sign = torch.where(_uni(g, rows.numel()) < 0.5, -1.0, 1.0)
        val = torch.exp(2.0 * val) * sign
        kind, a, b = _uni(g, n), _uni(g, n, -5.0, 0.0), _uni(g, n, 0.0, 5.0)
        boxed, free = (kind >= 0.5) & (kind < 0.8), kind >= 0.8
        inf = torch.full_like(a, math.inf)
        l = torch.where(boxed, a, torch.where(free, -inf, torch.zeros_like(a)))
        u = torch.where(boxed, b, inf)
    c, q, x = _plant(g, B, rows, cols, val, l, u)
    d = _finish(B, rows, cols, val, c, q, l, u)
    if case["qp"]:
        d.qd = torch.where(_uni(g, n) < 0.6, _uni(g, n, 0.0, 2.0), torch.zeros_like(c))
        d.c = c - d.qd * x
    return d


def _transport(case, seed, count):
    """Members of one transportation family (affine in a latent theta, plus
    noise) and start points near what a predictor returns: x and y of the
    right scale, off by noise."""
    g, S, T = _gen(seed, 2), case["sources"], case["sinks"]
    N, M = S * T, S + T
    fam = _gen(7, 3)  # the family itself is the same for every seed
    ps, pt = _uni(fam, (S, 2)), _uni(fam, (T, 2))
    c0 = ((ps[:, None] - pt[None]) ** 2).sum(-1).sqrt().flatten() * 10.0 + 1.0
    Cc = torch.randn(N, 16, dtype=F64, device="cuda", generator=fam) * 0.5
    s0, d0 = _uni(fam, S, 1.0, 3.0), _uni(fam, T, 1.0, 2.0)
    B = _blocks([M] * count, [N] * count, [T] * count)
    i = torch.arange(N, device="cuda")
    sink = torch.arange(T, device="cuda").repeat_interleave(S)
    cols1 = torch.cat([torch.arange(S, device="cuda").repeat(T) * T + sink, i])
    rows1 = torch.cat([sink, T + i // T])
    val1 = torch.cat([torch.ones(N, dtype=F64, device="cuda"), -torch.ones(N, dtype=F64, device="cuda")])
    shift = torch.arange(count, device="cuda")[:, None]
    rows, cols = (rows1[None] + shift * M).flatten(), (cols1[None] + shift * N).flatten()
    theta = torch.randn(count, 16, dtype=F64, device="cuda", generator=g)
    noise = lambda *s: 0.1 * torch.randn(*s, dtype=F64, device="cuda", generator=g)  # noqa: E731
    cost = c0[None] + (Cc[None] * theta[:, None, :]).sum(-1) + noise(count, N)
    s = (s0[None] * (1.0 + 0.3 * torch.tanh(theta[:, :1])) + noise(count, S)).clamp_(min=0.05)
    d = (d0[None] * (1.0 - 0.2 * torch.tanh(theta[:, 1:2])) + noise(count, T)).clamp_(min=0.05)
    s = s * (1.05 * d.sum(1, keepdim=True) / s.sum(1, keepdim=True))
    q = torch.cat([d, -s], 1).flatten()
    zero = torch.zeros(count * N, dtype=F64, device="cuda")
    lp = _finish(B, rows, cols, val1.repeat(count), cost.flatten(), q, zero, zero + math.inf)
    share = (s[:, :, None] * d[:, None, :] / s.sum(1)[:, None, None]).flatten()
    lp.x0 = share * (1.0 + 0.3 * torch.randn(count * N, dtype=F64, device="cuda", generator=g)).clamp_(min=0.0)
    lp.y0 = (torch.randn(count * M, dtype=F64, device="cuda", generator=g) + 2.0).abs()
    return lp


def _batch(case, seed):
    """Uneven planted LPs: m ~ logU, n ~ logU[2m/3, 2.5m], density U[0.5 %,
    5 %] (the shapes belong to the case), N(0, 1) values, 0 <= x <= 10."""
    rng = np.random.default_rng(case["shapes"])
    ms = np.rint(np.exp(rng.uniform(math.log(case["m_lo"]), math.log(case["m_hi"]), case["count"]))).astype(int)
    ns = np.rint(np.exp(rng.uniform(np.log(2 * ms / 3), np.log(2.5 * ms)))).astype(int)
    dens = rng.uniform(0.005, 0.05, case["count"])
    g = _gen(seed, 4)
    B = _blocks(ms, ns, ms // 2)
    p = torch.tensor(dens, device="cuda")[B.row_blk]
    lengths = torch.binomial(B.ns[B.row_blk].double(), p, generator=g).long().clamp_(min=1)
    rows, cols = _entries(g, B, lengths, True)
    val = torch.randn(rows.numel(), dtype=F64, device="cuda", generator=g)
    l, u = torch.zeros(B.N, dtype=F64, device="cuda"), torch.full((B.N,), 10.0, dtype=F64, device="cuda")
    c, q, _ = _plant(g, B, rows, cols, val, l, u)
    return _finish(B, rows, cols, val, c, q, l, u)


def _inputs(case, seed):
    kind = case["kind"]
    if kind in ("transport", "tbatch"):
        return _transport(case, seed, case.get("count", 1))
    return _batch(case, seed) if kind == "batch" else _lp(case, seed)


def _host_lps(d):
    """The blocks as separate host LPs."""
    h = {k: getattr(d, k).cpu().numpy() for k in ("ptr", "cols", "val", "c", "q", "l", "u")}
    ro, co, ne = d.B.ro.cpu().numpy(), d.B.co.cpu().numpy(), d.B.n_eqs.cpu().numpy()
    out = []
    for b in range(d.B.count):
        r0, r1, c0, c1 = ro[b], ro[b + 1], co[b], co[b + 1]
        e0, e1 = h["ptr"][r0], h["ptr"][r1]
        out.append(SimpleNamespace(m=int(r1 - r0), n=int(c1 - c0), n_eq=int(ne[b]), c=h["c"][c0:c1], q=h["q"][r0:r1],
                                   l=h["l"][c0:c1], u=h["u"][c0:c1], row_ptr=(h["ptr"][r0:r1 + 1] - e0).astype(np.int32),
                                   col_idx=(h["cols"][e0:e1] - c0).astype(np.int32), val=h["val"][e0:e1]))
    return out


def _mlp_data(case, seed):
    g = _gen(seed, 5)
    samples = 512 if case["kind"] == "train" else 64
    X = torch.randn(samples, 16, device="cuda", generator=g)
    mix = torch.randn(16, case["out"], device="cuda", generator=g) * 0.5
    T = torch.tanh(X @ mix) + 0.3 * torch.randn(samples, case["out"], device="cuda", generator=g)
    H, O = case["hidden"], case["out"]
    parts = []
    for fi, fo in ((16, H), (H, H), (H, O)):
        parts += [(torch.rand(fi * fo, device="cuda", generator=g) * 2 - 1) * math.sqrt(6.0 / fi), torch.zeros(fo, device="cuda")]
    d = SimpleNamespace(X=X, T=T, p=torch.cat(parts), H=H, O=O)
    if case["kind"] == "train":
        d.idx = torch.stack([torch.randperm(samples, device="cuda", generator=g)[: case["batch"]] for _ in range(case["steps"])])
    else:
        d.Z = torch.randn(case["count"], 16, device="cuda", generator=g)
    return d


def _matrix(case, seed):
    B = _blocks([case["m"]], [case["n"]], [0])
    rows, cols = _pattern(_gen(7, 6), dict(case, pattern="zipf"), B)  # the pattern belongs to the case
    g = _gen(seed, 6)
    val = torch.exp(2.0 * torch.randn(rows.numel(), dtype=F64, device="cuda", generator=g))
    val = val * torch.where(_uni(g, rows.numel()) < 0.5, -1.0, 1.0)
    order = torch.argsort(cols, stable=True)
    ptr = lambda i, k: torch.cat([i.new_zeros(1), torch.cumsum(torch.bincount(i, minlength=k), 0)]).int()  # noqa: E731
    return SimpleNamespace(rows=rows, cols=cols, val=val, order=order, kp=ptr(rows, B.M), ki=cols.int(), tp=ptr(cols, B.N),
                           ti=rows[order].int())


# ---------------------------------------------------------------- one pass


def prepare(case, seed):
    kind = case["kind"]
    s = SimpleNamespace(case=case, kind=kind)
    if kind == "lp":
        d = _lp(case, seed)
        s.keep = [t.contiguous() for t in (d.c, d.ptr.int(), d.cols.int(), d.val, d.q, d.l, d.u)]
        torch.cuda.synchronize()  # the library's stream is not torch's
        dev = dict(zip(("c", "row_ptr", "col_idx", "val", "q", "l", "u"), (t.data_ptr() for t in s.keep)))
        shape = SimpleNamespace(m=case["m"], n=case["n"], n_eq=int(d.B.n_eqs[0]), nnz=int(d.val.numel()),
                                qdiag=None if d.qd is None else d.qd.cpu().numpy())
        s.solver = P.Solver(shape, device=dev, value_bits=case["bits"])
        s.keep = None
    elif kind == "transport":
        d = _transport(case, seed, 1)
        s.solver = P.Solver(_host_lps(d)[0])
        s.x0, s.y0 = d.x0.cpu().numpy(), d.y0.cpu().numpy()
    elif kind in ("batch", "tbatch"):
        d = _inputs(case, seed)
        s.solver = P.BatchSolver(_host_lps(d))
        s.x0, s.y0 = (None, None) if d.x0 is None else (d.x0.cpu().numpy(), d.y0.cpu().numpy())
    elif kind in ("train", "predict"):
        d = _mlp_data(case, seed)
        s.net = P.Mlp(16, d.H, d.O, max_batch=case["max_batch"] if kind == "predict" else case["batch"])
        s.net.set_params(d.p.cpu().numpy())
        s.net.set_data(d.X.cpu().numpy(), d.T.cpu().numpy())
        if kind == "train":
            s.idx = d.idx.int().cpu().numpy()
        else:
            s.Z = d.Z.cpu().numpy()
    else:
        d = _matrix(case, seed)
        s.d, s.kv0, s.tv0 = d, d.val, d.val[d.order]
        s.kv, s.tv = torch.empty_like(s.kv0), torch.empty_like(s.tv0)
        s.D1 = torch.empty(case["m"], dtype=F64, device="cuda")
        s.D2 = torch.empty(case["n"], dtype=F64, device="cuda")
    return s


def run(s):
    case = s.case
    if s.kind == "lp":
        x, y, status, iters = s.solver.solve(tol=case["tol"], max_iter=case["iters"])
        return {"x": x, "y": y, "status": status, "iters": iters}
    if s.kind == "transport":
        x, y, status, iters = s.solver.solve(tol=case["tol"], max_iter=case["iters"], x0=s.x0, y0=s.y0)
        return {"x": x, "y": y, "status": status, "iters": iters}
    if s.kind in ("batch", "tbatch"):
        xs, ys, status, iters = s.solver.solve(tol=case["tol"], max_iter=case["iters"], x0=s.x0, y0=s.y0)
        return {"x": np.concatenate(xs), "y": np.concatenate(ys), "status": status, "iters": iters}
    if s.kind == "train":
        losses = s.net.train(s.idx, lr=1e-3)
        return {"losses": losses, "params": s.net.get_params()}
    if s.kind == "predict":
        return s.net.predict(s.Z)
    d = s.d
    s.kv.copy_(s.kv0)  # the entry point scales in place
    s.tv.copy_(s.tv0)
    P.pdlp_scale_device_noalloc(case["m"], case["n"], d.kp.data_ptr(), d.ki.data_ptr(), s.kv.data_ptr(), d.tp.data_ptr(),
                                d.ti.data_ptr(), s.tv.data_ptr(), 10, 1.0, s.D1.data_ptr(), s.D2.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
    return {"K": s.kv, "KT": s.tv, "D1": s.D1, "D2": s.D2}


# ---------------------------------------------------------------- necessary work


def work(case):
    """Operations of the algorithm; bytes of inputs and outputs once, and of
    the matrices and vectors in every iteration where they are too large to
    stay on the chip (128 MB)."""
    kind = case["kind"]
    if kind in ("lp", "transport", "batch", "tbatch"):
        if kind == "lp":
            M, N, Z = case["m"], case["n"], case["nnz"]
        elif kind == "batch":
            rng = np.random.default_rng(case["shapes"])
            ms = np.rint(np.exp(rng.uniform(math.log(case["m_lo"]), math.log(case["m_hi"]), case["count"])))
            ns = np.rint(np.exp(rng.uniform(np.log(2 * ms / 3), np.log(2.5 * ms))))
            M, N, Z = ms.sum(), ns.sum(), (ms * ns * rng.uniform(0.005, 0.05, case["count"])).sum()
        else:
            k = case.get("count", 1)
            M, N, Z = k * (case["sources"] + case["sinks"]), k * case["sources"] * case["sinks"], 2 * k * case["sources"] * case["sinks"]
        entry = 4 + case.get("bits", 64) // 8
        per_iter = 2 * entry * Z + 8 * (9 * N + 8 * M + (N if case.get("qp") else 0))
        once = per_iter + 8 * (N + M)
        return {"bytes": float(once if per_iter < 128e6 else per_iter * case["iters"]),
                "flops": float(case["iters"] * (4 * Z + 10 * N + 12 * M))}
    if kind in ("train", "predict"):
        H, O = case["hidden"], case["out"]
        params = 16 * H + H + H * H + H + H * O + O
        if kind == "predict":
            return {"bytes": 4.0 * (params + case["count"] * (16 + O)), "flops": 2.0 * case["count"] * params}
        # a step reads its targets once and reads and writes weights and both moments once
        per = 4.0 * case["batch"] * (16 + O) + 24.0 * params
        return {"bytes": case["steps"] * per + 4.0 * params, "flops": 6.0 * case["steps"] * case["batch"] * params}
    Z = case["nnz"]
    return {"bytes": 2.0 * 20 * Z + 8.0 * 2 * (case["m"] + case["n"]), "flops": 11.0 * 3 * Z}


# ---------------------------------------------------------------- in 64 bits, plain torch


def _scaled(rows, cols, val, M, N):
    """Ten Ruiz passes and one Pock-Chambolle pass: K~, D1, D2."""
    v, D1, D2 = val.clone(), torch.ones(M, dtype=F64, device="cuda"), torch.ones(N, dtype=F64, device="cuda")
    for it in range(11):
        a = v.abs()
        zr, zc = torch.zeros_like(D1), torch.zeros_like(D2)
        if it < 10:
            r, s = zr.scatter_reduce(0, rows, a, "amax"), zc.scatter_reduce(0, cols, a, "amax")
        else:
            r, s = zr.index_add(0, rows, a), zc.index_add(0, cols, a)
        r, s = (torch.where(t > 0, t.sqrt(), torch.ones_like(t)) for t in (r, s))
        v = v / r[rows] / s[cols]
        D1, D2 = D1 / r, D2 / s
    return v, D1, D2


def _csr(ptr, cols, val, shape):
    return torch.sparse_csr_tensor(ptr, cols, val, size=shape)


def _pdhg(d, case):
    """Restarted PDHG with adaptive steps on every block at once (one trial
    of each unfinished block per sweep)."""
    B, bits = d.B, case.get("bits", 64)
    M, N, rb, cb, iters, tol, period = B.M, B.N, B.row_blk, B.col_blk, case["iters"], case["tol"], 64
    v, D1, D2 = _scaled(d.rows, d.cols, d.val, M, N)
    order = torch.argsort(d.cols, stable=True)
    tptr = torch.cat([d.ptr.new_zeros(1), torch.cumsum(torch.bincount(d.cols, minlength=N), 0)])
    K64, T64 = _csr(d.ptr, d.cols, v, (M, N)), _csr(tptr, d.rows[order], v[order], (N, M))
    K, T = K64, T64
    if bits == 32:
        w = v.float().double()
        K, T = _csr(d.ptr, d.cols, w, (M, N)), _csr(tptr, d.rows[order], w[order], (N, M))
    c, q, l, u = D2 * d.c, D1 * d.q, d.l / D2, d.u / D2
    qd = None if d.qd is None else D2 * d.qd * D2
    one = B.count == 1
    sn = (lambda a: a.sum().reshape(1)) if one else (lambda a: _row_sums(a, B.ns))
    sm = (lambda a: a.sum().reshape(1)) if one else (lambda a: _row_sums(a, B.ms))
    ex = (lambda t: t) if one else (lambda t: t[cb])  # a block's scalar at its columns / rows
    ey = (lambda t: t) if one else (lambda t: t[rb])
    lf, uf = torch.isfinite(l), torch.isfinite(u)
    l_, u_ = torch.where(lf, l, torch.zeros_like(l)), torch.where(uf, u, torch.zeros_like(u))

    def pieces(x, y, Kx, KTy):
        rp = q - Kx
        rp = torch.where(B.ineq, rp.clamp(min=0), rp)
        grad = c if qd is None else c + qd * x
        dd = grad - KTy
        lam = torch.where(lf & uf, dd, torch.where(lf, dd.clamp(min=0), torch.where(uf, dd.clamp(max=0), torch.zeros_like(dd))))
        rd = dd - lam
        half = 0.0 if qd is None else 0.5 * sn(qd * x * x)
        pobj = sn(c * x) + half
        dobj = sm(q * y) + sn(l_ * lam.clamp(min=0) + u_ * lam.clamp(max=0)) - half
        return sm(rp * rp), sn(rd * rd), pobj, dobj, sm((rp / D1) ** 2).sqrt(), sn((rd / D2) ** 2).sqrt()

    def kkt(p, w):
        return (w * w * p[0] + p[1] / (w * w) + (p[3] - p[2]) ** 2).sqrt()

    qn, cn = sm(d.q * d.q).sqrt(), sn(d.c * d.c).sqrt()

    def rel(p):
        return torch.maximum((p[3] - p[2]).abs() / (1 + p[2].abs() + p[3].abs()), torch.maximum(p[4] / (1 + qn), p[5] / (1 + cn)))

    vmax = torch.zeros(B.count, dtype=F64, device="cuda").scatter_reduce(0, rb[d.rows], v.abs(), "amax")
    eta = 1.0 / vmax
    om = sn(c * c).sqrt() / sm(q * q).sqrt()
    x = torch.zeros(N, dtype=F64, device="cuda") if d.x0 is None else d.x0 / D2
    y = torch.zeros(M, dtype=F64, device="cuda") if d.y0 is None else d.y0 / D1
    Kx, g = K64 @ x, T64 @ y
    xl, yl, sx, sy = x.clone(), y.clone(), torch.zeros_like(x), torch.zeros_like(y)
    start = kkt(pieces(x, y, Kx, g), om)
    prev = start.clone()
    W, k, t = torch.zeros_like(eta), torch.zeros_like(eta), torch.zeros_like(eta)
    live = torch.ones_like(eta, dtype=torch.bool)
    status, best, stall = torch.ones(B.count, dtype=torch.int64, device="cuda"), math.inf, 0
    xo, yo, ko = x.clone(), y.clone(), k.clone()
    while bool(live.any()):
        tau, sig = ex(eta / om), ey(eta * om)
        xn = x - tau * (c - g)
        xn = torch.minimum(torch.maximum(xn if qd is None else xn / (1 + tau * qd), l), u)
        Kn = K @ xn
        yn = y + sig * (q - (2 * Kn - Kx))
        yn = torch.where(B.ineq, yn.clamp(min=0), yn)
        dx, dy = xn - x, yn - y
        dx2, dy2, cross = sn(dx * dx), sm(dy * dy), sm(dy * (Kn - Kx)).abs()
        bar = torch.where(cross > 0, (om * dx2 + dy2 / om) / (2 * cross), torch.full_like(cross, math.inf))
        nxt = torch.minimum((1 - (k + 2) ** -0.3) * bar, (1 + (k + 2) ** -0.6) * eta)
        acc = live & (eta <= bar)
        ax, ay = ex(acc), ey(acc)
        xp, x, y, Kx = x, torch.where(ax, xn, x), torch.where(ay, yn, y), torch.where(ay, Kn, Kx)
        sx, sy = torch.where(ax, sx + ex(eta) * xn, sx), torch.where(ay, sy + ey(eta) * yn, sy)
        W = torch.where(acc, W + eta, W)
        k, t = k + acc, t + acc
        eta = torch.where(live, nxt, eta)
        g = torch.where(ax, T @ y, g)
        due = acc & ((k % period == 0) | (k >= iters))
        if not bool(due.any()):
            continue
        dx_, dy_ = ex(due), ey(due)
        g = torch.where(dx_, T64 @ y, g)
        xb, yb = sx / ex(W), sy / ey(W)
        Kb, gb = K64 @ xb, T64 @ yb
        pc, pa = pieces(x, y, Kx, g), pieces(xb, yb, Kb, gb)
        okc, oka = rel(pc) <= tol, rel(pa) <= tol
        end = due & (okc | oka | (k >= iters))
        avg = end & ~okc & oka
        status = torch.where(end & (okc | oka), torch.zeros_like(status), status)
        fx, fy, wx, wy = ex(end), ey(end), ex(avg), ey(avg)
        xo, yo = torch.where(fx, torch.where(wx, xb, x), xo), torch.where(fy, torch.where(wy, yb, y), yo)
        ko = torch.where(end, k, ko)
        live = live & ~end
        kc, ka = kkt(pc, om), kkt(pa, om)
        ca = ~(kc < ka)
        kb = torch.where(ca, ka, kc)
        rs = due & ~end & ((kb <= 0.2 * start) | ((kb <= 0.8 * start) & (kb > prev)) | (t >= 0.36 * k))
        prev = torch.where(due & ~end, kb, prev)
        if not bool(rs.any()):
            continue
        if bits == 32 and K is not K64:
            now = float((rel(pa) if bool(ca[0]) else rel(pc))[0])
            best, stall = (now, 0) if now < best else (best, stall + 1)
            if stall >= 2:
                K, T = K64, T64
        mx, my, rx, ry = ex(rs & ca), ey(rs & ca), ex(rs), ey(rs)
        x, g, y, Kx = torch.where(mx, xb, x), torch.where(mx, gb, g), torch.where(my, yb, y), torch.where(my, Kb, Kx)
        dxn, dyn = sn((x - xl) ** 2).sqrt(), sm((y - yl) ** 2).sqrt()
        om = torch.where(rs & (dxn > 1e-10) & (dyn > 1e-10), torch.exp(0.5 * torch.log(dyn / dxn) + 0.5 * torch.log(om)), om)
        xl, yl = torch.where(rx, x, xl), torch.where(ry, y, yl)
        sx, sy = torch.where(rx, torch.zeros_like(sx), sx), torch.where(ry, torch.zeros_like(sy), sy)
        W, t = torch.where(rs, torch.zeros_like(W), W), torch.where(rs, torch.zeros_like(t), t)
        again = torch.where(ca, kkt(pa, om), kkt(pc, om))
        start, prev = torch.where(rs, again, start), torch.where(rs, again, prev)
    return torch.minimum(torch.maximum(D2 * xo, d.l), d.u), D1 * yo


def _net(p, H, O):
    out, at = [], 0
    for fi, fo in ((16, H), (H, H), (H, O)):
        out += [p[at:at + fi * fo].view(fi, fo), p[at + fi * fo:at + fi * fo + fo]]
        at += fi * fo + fo
    return out


def _forward(w, X):
    h1 = (X @ w[0] + w[1]).clamp(min=0)
    h2 = (h1 @ w[2] + w[3]).clamp(min=0)
    return h1, h2, h2 @ w[4] + w[5]


def exact(case, seed):
    kind = case["kind"]
    if kind in ("lp", "transport", "batch", "tbatch"):
        x, y = _pdhg(_inputs(case, seed), case)
        return {"x": x, "y": y, "status": None, "iters": None}
    if kind == "scale":
        d = _matrix(case, seed)
        v, D1, D2 = _scaled(d.rows, d.cols, d.val, case["m"], case["n"])
        return {"K": v, "KT": v[d.order], "D1": D1, "D2": D2}
    d = _mlp_data(case, seed)
    p, X, T = d.p.double(), d.X.double(), d.T.double()
    mu, sd = T.mean(0), T.std(0, unbiased=False).clamp(min=1e-6)
    if kind == "predict":
        return _forward(_net(p, d.H, d.O), d.Z.double())[2] * sd + mu
    m1, m2, losses = torch.zeros_like(p), torch.zeros_like(p), []
    for step, idx in enumerate(d.idx, 1):
        w = _net(p, d.H, d.O)
        x = X[idx]
        h1, h2, out = _forward(w, x)
        e = out - (T[idx] - mu) / sd
        losses.append((e * e).mean())
        dy = 2.0 * e / e.numel()
        d2 = (dy @ w[4].T) * (h2 > 0)
        d1 = (d2 @ w[2].T) * (h1 > 0)
        grad = torch.cat([(x.T @ d1).flatten(), d1.sum(0), (h1.T @ d2).flatten(), d2.sum(0), (h2.T @ dy).flatten(), dy.sum(0)])
        m1, m2 = 0.9 * m1 + 0.1 * grad, 0.999 * m2 + 0.001 * grad * grad
        p = p - 1e-3 * (m1 / (1 - 0.9 ** step)) / ((m2 / (1 - 0.999 ** step)).sqrt() + 1e-8)
    return {"losses": torch.stack(losses), "params": p}
