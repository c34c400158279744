"""Explicit bounds around the sizes of the tables that the partition's kernels
keep in shared memory: a full table up to 512 blocks, the bounds alone up to
5,120 of them, neither beyond. Counts, means and cells are the oracle's to the
bit, in the float32 cells, the planes and the bf16 cells."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402


def grid(rng, size, parts):
    """Bounds with empty and long blocks among them, and a permutation."""
    b = np.sort(rng.integers(0, size + 1, parts - 1))
    return (np.concatenate([[0], b, [size]]).astype(np.int64),
            rng.permutation(size).astype(np.int32))


@pytest.mark.parametrize("p,q", [(32, 16), (513, 1), (1, 513), (27, 19),
                                 (64, 40), (2, 2600), (5116, 2), (5117, 2)])
@pytest.mark.parametrize("equal", ["", "rows", "columns"])
def test_blocks_of_explicit_bounds(p, q, equal):
    rng = np.random.default_rng(p + q)
    m, n, nnz = 5300, 2700, 40000
    cells = np.unique(rng.integers(0, m * n, nnz))
    rng.shuffle(cells)
    u, i = (a.astype(np.int32) for a in np.divmod(cells, n))
    kw = {}
    if equal != "rows":
        kw["row_bounds"], kw["row_perm"] = grid(rng, m, p)
    if equal != "columns":
        kw["col_bounds"], kw["col_perm"] = grid(rng, n, q)
    stars = rng.integers(1, 6, len(u)).astype(np.float32)
    for x, prec in ((stars, bs.FP32), (stars + np.float32(0.25) * (u % 2 > 0),
                                       bs.FP32), (stars, bs.BF16)):
        part = oracle.partition(m, n, u, i, x, p, q, **kw)
        with bs.Context(precision=prec) as ctx:
            ctx.partition(m, n, u, i, x, p, q, **kw)
            cnt, mu = ctx.block_stats()
            assert np.array_equal(cnt, part.counts)
            assert np.array_equal(mu, part.mu32)
            busy = np.argsort(-cnt)[[0, 1, min(5, p * q - 1), p * q // 3]]
            for b in busy.tolist():
                got = ctx.get_block(b, want_factors=False,
                                    want_dense=True)["dense"]
                want = oracle.dense_block(part, b, fp32=True)
                if prec == bs.BF16:
                    want = torch.from_numpy(np.float32(want)).bfloat16().float()
                assert np.array_equal(got, np.asarray(want)), b


@pytest.mark.parametrize("p,q", [(128, 64), (8193, 1), (91, 91)])
def test_means_of_many_empty_blocks(p, q):
    """Around 8,192 blocks, where the mean of all ratings is taken once."""
    rng = np.random.default_rng(p)
    m, n = 9000, 100
    u = rng.integers(0, m, 3000).astype(np.int32)
    i = ((u * 7 + rng.integers(0, 3, 3000)) % n).astype(np.int32)
    x = rng.integers(1, 11, 3000).astype(np.float32) / 2
    part = oracle.partition(m, n, u, i, x, p, q)
    assert (part.counts == 0).any()
    for kw in ({}, dict(gram_path=1)):
        with bs.Context(**kw) as ctx:
            ctx.partition(m, n, u, i, x, p, q)
            cnt, mu = ctx.block_stats()
            assert np.array_equal(cnt, part.counts)
            assert np.array_equal(mu, part.mu32)
