"""Planes of 256 MB and more, which the partition fills chunk by chunk: every
cell against the ratings, bit for bit, over uneven blocks of both
orientations, permutations, ratings sorted by cell and shuffled, blocks
without a rating, a chunk with a rating in every cell, and held blocks only."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402


@pytest.mark.parametrize("precision,m,n", [(bs.FP32, 21007, 3601),
                                           (bs.FP32, 3601, 21007),
                                           (bs.BF16, 13001, 11003)])
@pytest.mark.parametrize("order,scale", [("sorted", 1.0), ("shuffled", 0.5)])
def test_every_cell(precision, m, n, order, scale):
    rng = np.random.default_rng(m + len(order))
    nnz = 300000
    cells = np.unique(rng.integers(0, m * n, nnz))
    cells = cells[(cells // n < 600) | (cells // n >= 700)]   # empty blocks
    full = (1500 + np.arange(70))[:, None] * n + np.arange(900)
    cells = np.union1d(cells, full)             # dense rows: whole chunks
    if order == "shuffled":
        cells = rng.permutation(cells)
    u, i = (cells // n).astype(np.int32), (cells % n).astype(np.int32)
    x = (rng.integers(1, 11, len(u)) * scale).astype(np.float32)
    rb = np.array([0, 600, 700, m // 2 + 1, m], np.int64)
    cb = np.array([0, 33, n // 3, n], np.int64)
    rp, cp = np.arange(m, dtype=np.int32), np.arange(n, dtype=np.int32)
    if order == "shuffled":
        cp = rng.permutation(n).astype(np.int32)
    owned = np.ones(12, np.int32)
    owned[[0, 5]] = 0
    with bs.Context(precision=precision) as ctx:
        ctx.set_owned(owned if order == "shuffled" else None)
        ctx.partition(m, n, u, i, x, 4, 3, rb, cb, rp, cp)
        cnt, mu = ctx.block_stats()
        W = np.zeros((m, n), np.float32)
        bi = np.searchsorted(rb, u, side="right") - 1
        bj = np.searchsorted(cb, cp[i], side="right") - 1
        assert np.array_equal(cnt, np.bincount(3 * bi + bj, minlength=12))
        y = torch.from_numpy(x - mu[3 * bi + bj])
        if precision == bs.BF16:
            y = y.bfloat16().float()
        W[u, cp[i]] = y.numpy()
        for b in range(12):
            if order == "shuffled" and not owned[b]:
                continue
            got = ctx.get_block(b, want_factors=False, want_dense=True)["dense"]
            p, q = divmod(b, 3)
            assert np.array_equal(got, W[rb[p]:rb[p + 1], cb[q]:cb[q + 1]]), b
