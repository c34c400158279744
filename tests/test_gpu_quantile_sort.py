"""The activity order around the sizes where its sort changes (one CTA's tile
of 4,096 ids, tiles of the radix sort), with few ratings (one pass) and more
than 2^16 (three), ties everywhere and one id holding most ratings."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402


@pytest.mark.parametrize("size", [1, 31, 4095, 4096, 4097, 8192, 8193, 70001])
@pytest.mark.parametrize("nnz", [0, 200, 300000])
def test_order_and_bounds(size, nnz):
    rng = np.random.default_rng(size + nnz)
    u = rng.integers(0, size, nnz).astype(np.int32)
    u[: nnz // 2] = size // 3                   # one busy id, the rest tie
    i = np.minimum(rng.geometric(0.01, nnz), 500).astype(np.int32) - 1
    p = min(size, 7)
    with bs.Context() as ctx:
        kw = ctx.quantile_grid(size, 500, u, i, p, 3)
    for ids, n, parts, side in ((u, size, p, "row"), (i, 500, 3, "col")):
        perm, bounds = oracle.activity_quantile_cut(ids, n, parts)
        assert np.array_equal(kw[side + "_perm"], perm)
        assert np.array_equal(kw[side + "_bounds"], bounds)
