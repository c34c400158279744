"""The radix sort around the number of 4,096-key tiles (16) up to which the
scatter adds up the tiles' counts itself: the quantile grid's sort of ids and
the blocked SGD's sorts of ratings, against the oracle's orders."""
import numpy as np
import pytest

import oracle
import synth
from oracle import sgd as osgd

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402


@pytest.mark.parametrize("size", [8192, 65535, 65536, 65537, 73728])
def test_quantile_order_of_many_ids(size):
    rng = np.random.default_rng(size)
    n = 50
    u = (size * rng.random(3 * size) ** 3).astype(np.int32)
    i = rng.integers(0, n, 3 * size).astype(np.int32)
    with bs.Context() as ctx:
        got = ctx.quantile_grid(size, n, u, i, 6, 3)
    for ids, count, parts, side in ((u, size, 6, "row"), (i, n, 3, "col")):
        perm, bounds = oracle.activity_quantile_cut(ids, count, parts)
        assert np.array_equal(got[side + "_perm"], perm)
        assert np.array_equal(got[side + "_bounds"], bounds)


@pytest.mark.parametrize("nnz", [4096, 4097, 65536, 65537])
def test_epoch_order_of_many_ratings(nnz):
    m, n, k = 700, 900, 4
    rng = np.random.default_rng(nnz)
    cells = rng.permutation(m * n)[:nnz]
    u, i = (a.astype(np.int32) for a in np.divmod(cells, n))
    x = rng.integers(1, 6, nnz).astype(np.float32)
    P0, Q0 = synth.sgd_start(m, n, k, 7)
    with bs.Context() as ctx:
        ctx.partition(m, n, u, i, x, 5, 3)
        ctx.sgd_prepare(u, i, x)
        ctx.sgd_train(P0, Q0, max_steps=1, delta=-1e300)
        got = ctx.sgd_get()
    ref = osgd.train(oracle.make_grid(m, n, 5, 3), u, i, x, P0, Q0, 1,
                     delta=-1e300)
    for a, b in zip(got, (ref.P, ref.Q, ref.bu, ref.bi)):
        assert np.array_equal(a, b)
