"""The prediction's forms (lanes per query by their number, the grid's table
from 250,001 queries on) and the squared errors' two, around the sizes where
one follows the other: the same bits as a short call's, which
test_gpu_predict.py compares with float64, and those sums' error against
float64 directly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402

# as in test_gpu_predict.py: at most 57 products and the mean in float32
REL = (2 * 57 + 4) * 2.0 ** -24


def fitted(p, q, k, quantile, seed=9):
    rng = np.random.default_rng(seed + k)
    m, n, nnz = 1300, 700, 30000
    cells = rng.permutation(m * n)[:nnz]
    u, i = (cells // n).astype(np.int32), (cells % n).astype(np.int32)
    x = rng.integers(1, 6, nnz).astype(np.float32)
    ctx = bs.Context()
    if quantile:
        kw = ctx.quantile_grid(m, n, u, i, p, q)
        ctx.partition(m, n, u, i, x, p, q, **kw)
    else:
        br, bc = -(-m // p), -(-n // q)
        kw = dict(row_bounds=np.minimum(np.arange(p + 1) * br, m),
                  col_bounds=np.minimum(np.arange(q + 1) * bc, n),
                  row_perm=np.arange(m), col_perm=np.arange(n))
        ctx.partition(m, n, u, i, x, p, q)
    ctx.factor(k, warn=False)
    return ctx, rng, m, n, kw


def exact(ctx, kw, q, u, i):
    """Predictions in float64 and the magnitudes that went into them."""
    r, c = kw["row_perm"][u], kw["col_perm"][i]
    bi = np.searchsorted(kw["row_bounds"][1:-1], r, side="right")
    bj = np.searchsorted(kw["col_bounds"][1:-1], c, side="right")
    y, mag = np.empty(len(u)), np.empty(len(u))
    blk = bi * q + bj
    for b in np.unique(blk):
        at = blk == b
        g = ctx.get_block(int(b))
        P = g["P"][(r - kw["row_bounds"][bi])[at]].astype(np.float64)
        V = g["V"][(c - kw["col_bounds"][bj])[at]].astype(np.float64)
        y[at] = float(g["mu"]) + (P * V).sum(1)
        mag[at] = abs(float(g["mu"])) + np.abs(P * V).sum(1)
    return y, mag


# two chunks a row or fewer, up to five, more; four sums and eight; grids with
# a table, with the bounds alone, and equal ones
@pytest.mark.parametrize("k", [3, 7, 11, 19, 32, 40, 56])
@pytest.mark.parametrize("p,q,quantile", [(3, 2, False), (3, 2, True),
                                          (32, 16, True), (27, 19, True),
                                          (27, 19, False)])
def test_forms_agree_around_their_sizes(k, p, q, quantile):
    ctx, rng, m, n, kw = fitted(p, q, k, quantile)
    with ctx:
        N = 500100
        qu = rng.integers(0, m, N).astype(np.int32)
        qi = rng.integers(0, n, N).astype(np.int32)
        du, di = torch.from_numpy(qu).cuda(), torch.from_numpy(qi).cuda()
        many = ctx.predict(du, di, out=torch.empty(N, device="cuda"))
        for nq in (1, 25000, 25001, 50001, 100001, 200001, 250000, 250001):
            y = ctx.predict(du[:nq], di[:nq], out=torch.empty(nq, device="cuda"))
            assert torch.equal(y, many[:nq]), nq
        at = np.concatenate([np.arange(300), rng.integers(0, N, 700)])
        y, mag = exact(ctx, kw, q, qu[at], qi[at])
        got = many.cpu().numpy().astype(np.float64)
        assert np.all(np.abs(got[at] - y) <= REL * mag + 1e-30)
        # the sum of N squares in float64, in any order
        t = torch.from_numpy(rng.uniform(1, 5, N).astype(np.float32)).cuda()
        d2 = (got - t.cpu().numpy().astype(np.float64)) ** 2
        for nq in (1, 31, 77824, 77825, 100000, 100001, 130001, N):
            s, cnt = ctx.sqerr(du[:nq], di[:nq], t[:nq])
            assert cnt == nq
            assert abs(s - d2[:nq].sum()) <= nq * 2.0 ** -52 * d2[:nq].sum()
        # an id out of range at the end of the long form is reported
        qu[-1] = m
        with pytest.raises(bs.BsvdError):
            ctx.predict(torch.from_numpy(qu).cuda(), di,
                        out=torch.empty(N, device="cuda"))
        with pytest.raises(bs.BsvdError):
            ctx.sqerr(torch.from_numpy(qu).cuda(), di, t)
