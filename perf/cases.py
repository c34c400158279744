"""The calls whose time is kept track of, through the library's public entry points.

Each case is one kind of call at one size. `listed()` holds the ones that are
looked at by name, `draw()` gives others of the same ranges. Ratings follow
the shapes of the synthetic workloads (long-tailed user and item activity, a
low-rank taste model plus noise) but are drawn on the GPU, from a seed.

Kinds:
  stats        block counts and means into preallocated arrays
  fit          partition, factorise and predict the held-out ratings
  partition    the activity-quantile grid and the partition on it
  factor       factorise an existing partition and predict the held-out ratings
  served       one batch of the server: host requests in, host predictions out
  predict      predictions of many ratings from fitted factors
  reconstruct  the dense rank-k matrix of one block
  sgd          the blocked SGD: epoch order, epochs, and the model read back
"""
import math

import numpy as np
import torch

import paper_1907_07410_gb300 as bs
from paper_1907_07410_gb300 import serve

PRECISION = {"fp32": bs.FP32, "tf32": bs.TF32, "bf16": bs.BF16}


def listed():
    return [
        # the smallest call: a caller with fixed memory asks for block means
        # of a MovieLens-100K-shaped matrix
        dict(name="stats_small", kind="stats", m=943, n=1682, nnz=90000,
             p=2, q=2),
        # a whole fit of the same matrix: launches and latency count
        dict(name="fit_small", kind="fit", m=943, n=1682, nnz=90000,
             held=10000, p=2, q=2, k=10, precision="fp32", scale="stars",
             grid="equal"),
        # a whole fit of a MovieLens-1M-shaped matrix, the ordinary size
        dict(name="fit_medium", kind="fit", m=6040, n=3952, nnz=900189,
             held=100020, p=4, q=4, k=20, precision="fp32", scale="stars",
             grid="equal"),
        # a whole fit of a Netflix-prize-shaped matrix in the form that the
        # batched workload names: the largest
        dict(name="fit_large_bf16", kind="fit", m=480189, n=17770,
             nnz=90432457, held=10048050, p=32, q=8, k=40, precision="bf16",
             scale="stars", grid="quantile"),
        # new ratings arrive: cut the grid again and lay the blocks out, for
        # the float32 form
        dict(name="partition_mid", kind="partition", m=120000, n=8000,
             nnz=10800000, p=16, q=4, precision="fp32", scale="stars"),
        # many small blocks of the medium matrix: a refit with another rank
        # or seed keeps its partition
        dict(name="factor_16x16_bf16", kind="factor", m=6040, n=3952,
             nnz=900189, held=100020, p=16, q=16, k=20, precision="bf16",
             scale="stars", grid="equal"),
        # ratings in half stars, on ragged sizes and uneven blocks, float32
        dict(name="factor_halfstars", kind="factor", m=20011, n=2999,
             nnz=1350007, held=149993, p=8, q=4, k=20, precision="fp32",
             scale="halves", grid="quantile"),
        # the server's batch of independent requests, host memory to host
        # memory
        dict(name="served_batch", kind="served", requests=16, rows_lo=128,
             rows_hi=8192, cols_lo=64, cols_hi=2048, queries=64),
        # scoring ten million candidates with a fitted model
        dict(name="predict_mid", kind="predict", m=120000, n=8000,
             nnz=10800000, held=10000001, p=16, q=4, k=40, precision="bf16",
             scale="stars", grid="quantile"),
        # a block's predictions for every cell, kept on the device; odd rows
        dict(name="reconstruct_large", kind="reconstruct", m=60013, n=4001,
             nnz=3000000, k=40, precision="bf16", scale="stars"),
        # the paper's own method in its own type, on its 8 x 8 grid
        dict(name="sgd_double_8x8", kind="sgd", m=6040, n=3952, nnz=900189,
             p=8, q=8, k=13, epochs=2, precision="fp64"),
        # the same in float32 on a fine grid
        dict(name="sgd_single_64x64", kind="sgd", m=6040, n=3952, nnz=900189,
             p=64, q=64, k=13, epochs=3, precision="fp32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _matrix(rng, m_lo, m_hi, n_lo, n_hi, nnz_hi):
    m, n = _log(rng, m_lo, m_hi), _log(rng, n_lo, n_hi)
    hi = min(nnz_hi, int(0.25 * m * n))
    return dict(m=m, n=n, nnz=_log(rng, max(hi // 40, 500), hi))


def draw(rng):
    kind = rng.choice(["stats", "fit", "fit", "partition", "factor", "factor",
                       "served", "predict", "reconstruct", "sgd", "sgd"])
    c = dict(kind=kind)
    if kind == "served":
        c.update(requests=rng.randint(1, 16), rows_lo=128,
                 rows_hi=_log(rng, 256, 8192), cols_lo=64,
                 cols_hi=_log(rng, 128, 2048), queries=rng.randint(8, 256))
        return c
    if kind == "stats":
        c.update(_matrix(rng, 100, 40000, 60, 8000, 4000000))
        c.update(p=rng.randint(1, 48), q=rng.randint(1, 48))
        return c
    if kind == "sgd":
        c.update(_matrix(rng, 600, 8000, 400, 5000, 900000))
        c.update(p=_log(rng, 8, 128), q=_log(rng, 8, 128),
                 k=rng.randint(3, 32), epochs=rng.randint(1, 2),
                 precision=rng.choice(["fp64", "fp32"]))
        return c
    if kind == "reconstruct":
        c.update(_matrix(rng, 300, 60000, 200, 4000, 3000000))
        c.update(k=rng.randint(4, 56), precision=rng.choice(["fp32", "bf16"]),
                 scale="stars")
        return c
    c.update(_matrix(rng, 400, 120000, 300, 8000, 10000000))
    c.update(p=rng.randint(1, 16), q=rng.randint(1, 12),
             precision=rng.choice(["fp32", "fp32", "bf16", "tf32"]),
             scale=rng.choice(["stars", "stars", "halves", "real"]))
    if kind == "partition":
        return c
    c.update(held=max(64, c["nnz"] // 9), k=rng.randint(5, 56),
             grid=rng.choice(["equal", "quantile"]))
    if kind == "predict":
        c.update(held=_log(rng, 1000, 10000000))
        c["held"] = min(c["held"], c["m"] * c["n"] // 4)
    return c


# ---- inputs ---------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 1907)
    return g


def _nodes(size):
    """Ranks 1 .. size in a few hundred groups: middle rank and group size."""
    edges = np.unique(np.round(np.geomspace(1, size + 1, 300)).astype(np.int64))
    return torch.from_numpy(0.5 * (edges[:-1] + edges[1:] - 1)), \
        torch.from_numpy((edges[1:] - edges[:-1]).astype(np.float64))


def _cells(g, m, n, want, s_user, s_item, floor=20.0):
    """`want` distinct (user, item) cells in random order: a cell is taken
    with a probability that grows with its user's and its item's weight
    (rank^-s over a random ranking) and saturates at one."""
    ru, cu = _nodes(m)
    ri, ci = _nodes(n)
    wu, wi = ru.double().pow(-s_user), ri.double().pow(-s_item)
    base = min(floor, 0.2 * want / m) / float((wi * ci).sum())
    lo, hi = 1e-12, 1e12
    for _ in range(80):                     # the scale that gives `want` cells
        t = math.sqrt(lo * hi)
        lam = torch.outer(t * wu + base, wi)
        got = float(((1 - torch.exp(-lam)) * torch.outer(cu, ci)).sum())
        lo, hi = (t, hi) if got < want else (lo, t)
    urank = torch.randperm(m, generator=g, device="cuda")
    irank = torch.randperm(n, generator=g, device="cuda")
    iw = (irank + 1).float().pow(-s_item)
    t = hi
    for _ in range(40):
        t *= 1.03
        uw = (t * (urank + 1).double().pow(-s_user) + base).float()
        rows = max(1, (1 << 26) // n)
        keys = []
        for a in range(0, m, rows):
            lam = torch.outer(uw[a:a + rows], iw)
            draw_ = torch.rand(lam.shape, generator=g, device="cuda")
            hit = draw_ < lam.neg_().expm1_().neg_()
            keys.append(hit.view(-1).nonzero().view(-1) + a * n)
        key = torch.cat(keys)
        if key.numel() >= want:
            break
    else:
        raise ValueError("too many ratings for the matrix")
    key = key[torch.randperm(key.numel(), generator=g, device="cuda")[:want]]
    return torch.div(key, n, rounding_mode="floor").int(), (key % n).int()


def _values(g, m, n, u, i, scale, d=20):
    """Ratings of the cells: taste model plus noise, on the scale's grid."""
    U = torch.randn((m, d), generator=g, device="cuda") * 0.3
    V = torch.randn((n, d), generator=g, device="cuda") * 0.3
    x = torch.randn(u.numel(), generator=g, device="cuda") * 0.8 + 3.5
    for a in range(0, u.numel(), 1 << 22):
        b = slice(a, a + (1 << 22))
        x[b] += (U[u[b].long()] * V[i[b].long()]).sum(1)
    if scale == "stars":
        return torch.floor(x + 0.5).clamp_(1, 5)
    if scale == "halves":
        return (torch.floor(2 * x + 0.5) / 2).clamp_(0.5, 5)
    return (4 * (x - 3.5)).clamp_(-10, 10)      # a continuous scale


def _ratings(case, seed):
    g = _generator(seed)
    m, n, nnz = case["m"], case["n"], case["nnz"]
    total = nnz + case.get("held", 0)
    u, i = _cells(g, m, n, total, 1.2 if m > 10000 else 1.0, 0.9)
    x = _values(g, m, n, u, i, case.get("scale", "stars"))
    return (u[:nnz].contiguous(), i[:nnz].contiguous(), x[:nnz].contiguous(),
            u[nnz:].contiguous(), i[nnz:].contiguous())


def _requests(case, seed):
    g = _generator(seed)
    rng = np.random.Generator(np.random.PCG64(int(seed) + 11))
    reqs = []
    for _ in range(case["requests"]):
        m = int(rng.integers(case["rows_lo"], case["rows_hi"] + 1))
        n = int(rng.integers(case["cols_lo"], case["cols_hi"] + 1))
        k = int(rng.choice([10, 20, 40]))
        dens = float(rng.uniform(0.03, 0.10))
        hit = torch.rand((m, n), generator=g, device="cuda") < dens
        key = hit.view(-1).nonzero().view(-1)
        key = key[torch.randperm(key.numel(), generator=g, device="cuda")]
        u = torch.div(key, n, rounding_mode="floor").int()
        i = (key % n).int()
        x = _values(g, m, n, u, i, "stars", 10)
        u, i, x = u.cpu().numpy(), i.cpu().numpy(), x.cpu().numpy()
        nq = min(case["queries"], len(u) // 2)
        reqs.append(serve.Request(m, n, k, u[nq:].copy(), i[nq:].copy(),
                                  x[nq:].copy(), u[:nq].copy(), i[:nq].copy()))
    return reqs


# ---- the calls --------------------------------------------------------------

def _partition(case, st):
    if case.get("grid", "equal") == "quantile":
        return st["ctx"].partition_quantile(case["m"], case["n"], st["u"],
                                            st["i"], st["x"], case["p"],
                                            case["q"])
    return st["ctx"].partition(case["m"], case["n"], st["u"], st["i"],
                               st["x"], case["p"], case["q"])


def prepare(case, seed):
    kind = case["kind"]
    st = dict(case=dict(case))
    if kind == "served":
        st["reqs"] = _requests(case, seed)
        st["ctx"] = bs.Context()
        return st
    st["u"], st["i"], st["x"], st["qu"], st["qi"] = _ratings(case, seed)
    if kind == "stats":
        nb = case["p"] * case["q"]
        st["counts"] = torch.zeros(nb, dtype=torch.int64, device="cuda")
        st["mu"] = torch.zeros(nb, dtype=torch.float32, device="cuda")
        st["stream"] = torch.cuda.current_stream().cuda_stream
        return st
    if kind == "sgd":
        st["ctx"] = bs.Context()
        _partition(case, st)
        rng = np.random.Generator(np.random.PCG64(int(seed) + 13))
        st["P0"] = rng.normal(0.0, 0.1, size=(case["m"], case["k"]))
        st["Q0"] = rng.normal(0.0, 0.1, size=(case["n"], case["k"]))
        return st
    st["ctx"] = bs.Context(precision=PRECISION[case["precision"]])
    if kind in ("fit", "factor", "predict"):
        st["y"] = torch.zeros(case["held"], dtype=torch.float32, device="cuda")
    if kind in ("factor", "predict"):
        _partition(case, st)
    if kind == "predict":
        st["ctx"].factor(case["k"], warn=False)
    if kind == "reconstruct":
        st["ctx"].partition(case["m"], case["n"], st["u"], st["i"], st["x"],
                            1, 1)
        st["ctx"].factor(case["k"], warn=False)
        st["out"] = torch.zeros((case["m"], case["n"]), dtype=torch.float32,
                                device="cuda")
    return st


def run(st):
    case = st["case"]
    kind, ctx = case["kind"], st.get("ctx")
    if kind == "stats":
        bs.bsvd_block_means_noalloc(case["m"], case["n"], st["u"], st["i"],
                                    st["x"], case["p"], case["q"],
                                    st["counts"], st["mu"],
                                    stream=st["stream"])
        return st["counts"], st["mu"]
    if kind == "fit":
        _partition(case, st)
        ctx.factor(case["k"], warn=False)
        return ctx.predict(st["qu"], st["qi"], out=st["y"])
    if kind == "partition":
        rb, cb = ctx.partition_quantile(case["m"], case["n"], st["u"],
                                        st["i"], st["x"], case["p"],
                                        case["q"])
        counts, mu = ctx.block_stats()
        return rb, cb, counts, mu
    if kind == "factor":
        ctx.factor(case["k"], warn=False)
        return ctx.predict(st["qu"], st["qi"], out=st["y"])
    if kind == "served":
        return serve.run_batch(ctx, st["reqs"])
    if kind == "predict":
        return ctx.predict(st["qu"], st["qi"], out=st["y"])
    if kind == "reconstruct":
        return ctx.reconstruct(0, out=st["out"])
    ctx.sgd_prepare(st["u"], st["i"], st["x"])
    hist, _ = ctx.sgd_train(st["P0"], st["Q0"], max_steps=case["epochs"],
                            delta=-1e300,
                            precision=(bs.SGD_FP64
                                       if case["precision"] == "fp64"
                                       else bs.SGD_FP32))
    return (hist,) + tuple(ctx.sgd_get())


def work(case):
    """Least bytes and operations of a pass: ratings and queries read once,
    results written once; for the dense blocks, the cells once in the form's
    type (they are what the factorisation works on), the Gram's distinct
    entries and the projection."""
    kind = case["kind"]
    if kind == "served":
        m = 0.5 * (case["rows_lo"] + case["rows_hi"])
        n = 0.5 * (case["cols_lo"] + case["cols_hi"])
        r, s = case["requests"], min(m, n)
        return {"bytes": r * (12 * 0.065 * m * n + 4 * m * n
                              + 12 * case["queries"]),
                "flops": r * (m * n * s + 2 * m * n * 23)}
    m, n, nnz = case["m"], case["n"], case["nnz"]
    if kind == "stats":
        return {"bytes": 12 * nnz + 12 * case["p"] * case["q"], "flops": nnz}
    if kind == "sgd":
        e, k = case["epochs"], case["k"]
        w = 8 if case["precision"] == "fp64" else 4
        return {"bytes": 12 * nnz * (e + 1) + 2 * w * (m + n) * (k + 1),
                "flops": e * nnz * (12 * k + 13)}
    if kind == "reconstruct":
        k = case["k"]
        return {"bytes": 4 * m * n + 4 * (m + n) * k, "flops": 2 * m * n * k}
    cell = 2 if case["precision"] == "bf16" else 4
    if kind == "partition":
        return {"bytes": 12 * nnz + cell * m * n, "flops": nnz}
    k, held = case["k"], case["held"]
    if kind == "predict":
        return {"bytes": 12 * held + 4 * k * (m + n), "flops": 2 * k * held}
    s = min(m / case["p"], n / case["q"])
    flops = m * n * s + 2 * m * n * k + 2 * k * held
    nbytes = cell * m * n + 12 * held + 4 * k * (m + n)
    if kind == "fit":
        nbytes += 12 * nnz
    return {"bytes": nbytes, "flops": flops}


# ---- the same in 64 bits ------------------------------------------------------

def _quantile_side(ids, size, parts):
    cnt = torch.bincount(ids.long(), minlength=size)
    order = torch.sort(cnt, descending=True, stable=True).indices
    pos = torch.empty_like(order)
    pos[order] = torch.arange(size, device=order.device)
    run_ = torch.cat([torch.zeros(1, dtype=torch.int64, device=order.device),
                      torch.cumsum(cnt[order], 0)]) * parts
    total = int(cnt.sum())
    b = [0]
    for gg in range(1, parts):
        b.append(int(torch.searchsorted(run_, gg * total)))
    return pos, np.array(b + [size], np.int64)


def _equal_side(size, parts):
    step = -(-size // parts)
    return torch.arange(size, device="cuda"), \
        np.minimum(np.arange(parts + 1, dtype=np.int64) * step, size)


def _grid(case, u, i, quantile):
    if quantile:
        rp, rb = _quantile_side(u, case["m"], case["p"])
        cp, cb = _quantile_side(i, case["n"], case["q"])
    else:
        rp, rb = _equal_side(case["m"], case["p"])
        cp, cb = _equal_side(case["n"], case["q"])
    return rp, rb, cp, cb


def _locate(gr, u, i, q):
    rp, rb, cp, cb = gr
    r, c = rp[u.long()], cp[i.long()]
    trb, tcb = torch.from_numpy(rb).cuda(), torch.from_numpy(cb).cuda()
    bi = torch.searchsorted(trb[1:-1].contiguous(), r, right=True)
    bj = torch.searchsorted(tcb[1:-1].contiguous(), c, right=True)
    return bi * q + bj, r - trb[bi], c - tcb[bj]


def _block_means(blk, x, nb):
    cnt = torch.bincount(blk, minlength=nb)
    tot = torch.zeros(nb, dtype=torch.float64, device="cuda")
    tot.index_add_(0, blk, x.double())
    every = float(x.double().sum()) / max(1, x.numel())
    return torch.where(cnt > 0, tot / cnt.clamp(min=1), every)


def _truncated(B, k):
    """Both factors of the best rank-k approximation of a dense block."""
    trans = B.shape[1] <= B.shape[0]
    W = B.T if trans else B
    k = min(k, W.shape[0])
    if k == 0:
        return None
    _, vec = torch.linalg.eigh(W @ W.T)
    Fs = vec[:, -k:]
    FL = W.T @ Fs
    return (FL, Fs) if trans else (Fs, FL)


def _fit_exact(m, n, u, i, x, qu, qi, ks, gr, p, q):
    blk, r, c = _locate(gr, u, i, q)
    mu = _block_means(blk, x, p * q)
    qb, qr, qc = _locate(gr, qu, qi, q)
    y = mu[qb].clone()
    rb, cb = gr[1], gr[3]
    for b in range(p * q):
        mb = int(rb[b // q + 1] - rb[b // q])
        nb = int(cb[b % q + 1] - cb[b % q])
        if mb == 0 or nb == 0:
            continue
        at = blk == b
        B = torch.zeros((mb, nb), dtype=torch.float64, device="cuda")
        B[r[at], c[at]] = x[at].double() - mu[b]
        f = _truncated(B, ks)
        if f is None:
            continue
        at = qb == b
        y[at] += (f[0][qr[at]] * f[1][qc[at]]).sum(1)
    return y


def _solve_cost(m, n, p, q):
    """Of the 64-bit eigenproblems of a grid, as if its blocks were equal."""
    mb, nb = m / p, n / q
    s = min(mb, nb)
    return p * q * (25 * s ** 3 + 2 * mb * nb * s)


def _sgd_exact(case, seed):
    u, i, x, _, _ = _ratings(case, seed)
    m, n, p, q, k = (case[a] for a in "mnpqk")
    gr = _grid(case, u, i, False)
    blk, r, c = (t.cpu().numpy() for t in _locate(gr, u, i, q))
    bi, bj = blk // q, blk % q
    step = (bi - bj) % p if p >= q else (bj - bi) % q
    lane = bj if p >= q else bi
    order = np.lexsort((c, r, lane, step))
    u, i = u.cpu().numpy()[order], i.cpu().numpy()[order]
    x = x.cpu().numpy()[order].astype(np.float64)
    rng = np.random.Generator(np.random.PCG64(int(seed) + 13))
    P = rng.normal(0.0, 0.1, size=(m, k))
    Q = rng.normal(0.0, 0.1, size=(n, k))
    bu, bi_ = np.zeros(m), np.zeros(n)

    def rmse():
        d = x - ((P[u] * Q[i]).sum(1) + bu[u] + bi_[i])
        return math.sqrt(float((d * d).mean()))

    hist = [rmse()]
    for _ in range(case["epochs"]):
        for a, b, v in zip(u.tolist(), i.tolist(), x.tolist()):
            pu, qi = P[a].copy(), Q[b].copy()
            e = v - bu[a] - bi_[b] - float(pu @ qi)
            bu[a] += 0.004 * (e - 0.019 * bu[a])
            bi_[b] += 0.013 * (e - 0.007 * bi_[b])
            P[a] = pu + 0.019 * (e * qi - 0.019 * pu)
            Q[b] = qi + 0.004 * (e * pu - 0.019 * qi)
        hist.append(rmse())
    return np.array(hist), P, Q, bu, bi_


def exact(case, seed):
    kind = case["kind"]
    if kind == "sgd":
        if case["nnz"] * case["epochs"] > 400000:
            return None
        return _sgd_exact(case, seed)
    if kind == "served":
        reqs = _requests(case, seed)
        out = []
        for rq in reqs:
            t = [torch.from_numpy(a).cuda() for a in (rq.r, rq.c, rq.x, rq.qr,
                                                      rq.qc)]
            gr = _grid(dict(m=rq.m, n=rq.n, p=1, q=1), t[0], t[1], False)
            out.append(_fit_exact(rq.m, rq.n, *t, rq.k, gr, 1, 1))
        return out
    m, n = case["m"], case["n"]
    p, q = case.get("p", 1), case.get("q", 1)
    if kind in ("fit", "factor", "predict", "reconstruct") and \
            _solve_cost(m, n, p, q) > 1.5e12:
        return None
    u, i, x, qu, qi = _ratings(case, seed)
    gr = _grid(dict(case, p=p, q=q), u, i, kind == "partition"
               or case.get("grid") == "quantile")
    blk, _, _ = _locate(gr, u, i, q)
    if kind == "stats":
        return None, _block_means(blk, x, p * q)
    if kind == "partition":
        return None, None, None, _block_means(blk, x, p * q)
    if kind == "reconstruct":
        mu = _block_means(blk, x, 1)[0]
        B = torch.zeros((m, n), dtype=torch.float64, device="cuda")
        B[u.long(), i.long()] = x.double() - mu
        a, b = _truncated(B, case["k"])
        return mu + a @ b.T
    return _fit_exact(m, n, u, i, x, qu, qi, case["k"], gr, p, q)
