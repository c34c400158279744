"""Predictions and squared errors against float64 dot products of the block's
own factors, across the rules that pick the lanes per query and the grid
table, and at the ends of warps and CTAs."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402

# a dot product of at most 56 terms in float32, and the mean: each operation
# rounds by 2^-24 of the running magnitude; P = F_s sigma and V = F_L / sigma
# round once more each on their way to the host
REL = (2 * 57 + 4) * 2.0 ** -24


def blocks_of(ctx, nb):
    return [ctx.get_block(b) for b in range(nb)]


def expect(blocks, blk, r, c):
    y = np.empty(len(blk))
    mag = np.empty(len(blk))
    for t, b in enumerate(blk):
        g = blocks[b]
        p = g["P"][r[t]].astype(np.float64)
        v = g["V"][c[t]].astype(np.float64)
        y[t] = float(g["mu"]) + p @ v
        mag[t] = abs(float(g["mu"])) + np.abs(p) @ np.abs(v)
    return y, mag


def check(ctx, nb, locate, u, i, dev=False):
    blocks = blocks_of(ctx, nb)
    if dev:
        du, di = torch.from_numpy(u).cuda(), torch.from_numpy(i).cuda()
        out = torch.empty(len(u), device="cuda")
        got = ctx.predict(du, di, out=out).cpu().numpy()
    else:
        got = ctx.predict(u, i)
    y, mag = expect(blocks, *locate(u, i))
    assert np.all(np.abs(got - y) <= REL * mag + 1e-30)
    t = np.random.default_rng(1).uniform(1, 5, len(u)).astype(np.float32)
    s, n = ctx.sqerr(u, i, t)
    assert n == len(u)
    want = np.sum((got.astype(np.float64) - t) ** 2)
    assert abs(s - want) <= 1e-5 * want


def equal_locate(m, n, p, q):
    br, bc = -(-m // p), -(-n // q)
    return lambda u, i: ((u // br) * q + i // bc, u % br, i % bc)


@pytest.mark.parametrize("k", [1, 4, 5, 16, 17, 32, 33, 48, 49, 56])
def test_ranks_across_the_lane_rule(k):
    m, n, p, q = 301, 203, 2, 2
    r = synth.random_ratings(61, m, n, 9000, 777)
    with bs.Context() as ctx:
        ctx.partition(m, n, r.u_train, r.i_train, r.x_train, p, q)
        ctx.factor(k, warn=False)
        check(ctx, p * q, equal_locate(m, n, p, q), r.u_test, r.i_test)


@pytest.mark.parametrize("nq", [1, 31, 32, 33, 255, 257, 1000])
def test_query_counts(nq):
    m, n = 90, 70
    r = synth.random_ratings(62, m, n, 2000, nq)
    with bs.Context() as ctx:
        ctx.partition(m, n, r.u_train, r.i_train, r.x_train, 3, 2)
        ctx.factor(5, warn=False)
        check(ctx, 6, equal_locate(m, n, 3, 2), r.u_test, r.i_test, dev=True)


# 512 blocks and 512 block rows fit the table, one more of either does not
@pytest.mark.parametrize("p,q", [(32, 16), (27, 19), (512, 1), (513, 1),
                                 (1, 513)])
def test_grids_around_the_table_limit(p, q):
    m, n = 1200, 1100
    r = synth.random_ratings(63, m, n, 30000, 500)
    with bs.Context() as ctx:
        ctx.partition(m, n, r.u_train, r.i_train, r.x_train, p, q)
        ctx.factor(2, warn=False)
        check(ctx, p * q, equal_locate(m, n, p, q), r.u_test, r.i_test)


def test_uneven_bounds_with_permutations_and_empty_blocks():
    m, n = 200, 150
    r = synth.random_ratings(64, m, n, 8000, 600)
    rng = np.random.default_rng(3)
    rp = rng.permutation(m).astype(np.int32)
    cp = rng.permutation(n).astype(np.int32)
    rb = np.array([0, 50, 50, 130, 200], np.int64)
    cb = np.array([0, 20, 150], np.int64)

    def locate(u, i):
        a, c = rp[u], cp[i]
        bi = np.searchsorted(rb[1:-1], a, side="right")
        bj = np.searchsorted(cb[1:-1], c, side="right")
        return bi * 2 + bj, a - rb[bi], c - cb[bj]

    with bs.Context() as ctx:
        ctx.partition(m, n, r.u_train, r.i_train, r.x_train, 4, 2,
                      row_bounds=rb, col_bounds=cb, row_perm=rp, col_perm=cp)
        ctx.factor(9, warn=False)
        check(ctx, 8, locate, r.u_test, r.i_test)


def test_block_diagonal_and_ids_off_it():
    rb = np.array([0, 40, 70], np.int64)
    cb = np.array([0, 25, 60], np.int64)
    rng = np.random.default_rng(4)
    u = np.concatenate([rng.integers(0, 40, 300), rng.integers(40, 70, 300)])
    i = np.concatenate([rng.integers(0, 25, 300), rng.integers(25, 60, 300)])
    key = np.unique(u * 60 + i)
    u, i = (key // 60).astype(np.int32), (key % 60).astype(np.int32)
    x = rng.integers(1, 6, len(u)).astype(np.float32)

    def locate(a, c):
        b = (a >= 40).astype(int)
        return b, a - rb[b], c - cb[b]

    with bs.Context() as ctx:
        ctx.partition_diag(rb, cb, u, i, x)
        ctx.factor([3, 6], warn=False)
        check(ctx, 2, locate, u, i)
        for bad_u, bad_i in ((0, 30), (70, 0), (0, -1)):
            with pytest.raises(bs.BsvdError) as e:
                ctx.predict(np.array([1, bad_u], np.int32),
                            np.array([1, bad_i], np.int32))
            assert e.value.status == bs.EINVAL


def test_squared_errors_skip_blocks_of_another_shard():
    m, n = 120, 80
    r = synth.random_ratings(65, m, n, 3000, 700)
    owned = np.array([1, 0, 1, 0], np.uint8)
    blk = equal_locate(m, n, 2, 2)(r.u_test, r.i_test)[0]
    mine = owned[blk] == 1
    with bs.Context() as ctx:
        ctx.set_owned(owned)
        ctx.partition(m, n, r.u_train, r.i_train, r.x_train, 2, 2)
        ctx.factor(6, warn=False)
        s, cnt = ctx.sqerr(r.u_test, r.i_test, r.x_test)
        y = ctx.predict(r.u_test, r.i_test).astype(np.float64)
        mu = ctx.block_stats()[1]
    assert cnt == mine.sum()
    assert np.array_equal(y[~mine].astype(np.float32), mu[blk[~mine]])
    want = np.sum((y[mine] - r.x_test[mine]) ** 2)
    assert abs(s - want) <= 1e-12 * want


@pytest.mark.parametrize("k", [3, 10, 20, 40, 56])
@pytest.mark.parametrize("grid", ["equal", "quantile", "diag"])
def test_few_queries_equal_many(k, grid):
    """A short call takes the form with several lanes per query from the ids
    on; its sums are those of the long call, bit for bit."""
    rng = np.random.default_rng(k)
    m, n, nnz = 700, 300, 9000
    cells = rng.permutation(m * n)[:nnz]
    u, i = (cells // n).astype(np.int32), (cells % n).astype(np.int32)
    x = rng.integers(1, 6, nnz).astype(np.float32)
    with bs.Context() as ctx:
        if grid == "quantile":
            ctx.partition_quantile(m, n, u, i, x, 3, 2)
        elif grid == "equal":
            ctx.partition(m, n, u, i, x, 3, 2)
        else:
            keep = (u < 400) == (i < 100)
            ctx.partition_diag([0, 400, 700], [0, 100, 300], u[keep], i[keep],
                               x[keep])
        ctx.factor(k, warn=False)
        q = rng.integers(0, m * n, 40001 + 37)
        qu, qi = (q // n).astype(np.int32), (q % n).astype(np.int32)
        if grid == "diag":
            qi = np.where(qu < 400, qi % 100, 100 + qi % 200).astype(np.int32)
        many = ctx.predict(qu, qi)
        for nq in (1, 3, 4, 5, 31, 33, 1000, 40000):
            assert np.array_equal(ctx.predict(qu[:nq], qi[:nq]), many[:nq]), nq
        with pytest.raises(bs.BsvdError):
            ctx.predict(np.array([0, m], np.int32), np.array([0, 0], np.int32))
