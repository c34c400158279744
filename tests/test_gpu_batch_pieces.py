"""A batch partitioned from each matrix's own arrays against the same batch
stacked by the caller: empty pieces, pieces that begin at odd places, ids
outside the matrix. The same kernels run on the same ratings in the same
order, so everything is equal to the bit."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402
from paper_1907_07410_gb300 import serve  # noqa: E402


def matrices(sizes, seed):
    rng = np.random.default_rng(seed)
    us, is_, xs = [], [], []
    for m, n, nnz in sizes:
        cells = rng.permutation(m * n)[:nnz]
        us.append((cells // n).astype(np.int32))
        is_.append((cells % n).astype(np.int32))
        xs.append(rng.integers(1, 6, nnz).astype(np.float32))
    bounds = [np.concatenate([[0], np.cumsum([s[d] for s in sizes])])
              for d in (0, 1)]
    return bounds[0], bounds[1], us, is_, xs


@pytest.mark.parametrize("sizes", [
    [(5, 7, 11)],
    [(40, 30, 333), (1, 1, 1), (64, 3, 0), (129, 65, 4097), (33, 200, 5)],
    [(20 + b, 31 - b % 7, 1 + 13 * b % 97) for b in range(70)],
])
@pytest.mark.parametrize("device", [False, True])
def test_pieces_equal_the_stacked_batch(sizes, device):
    rb, cb, us, is_, xs = matrices(sizes, len(sizes))
    u = np.concatenate([a + np.int32(o) for a, o in zip(us, rb)])
    i = np.concatenate([a + np.int32(o) for a, o in zip(is_, cb)])
    got, want = bs.Context(), bs.Context()
    put = (lambda a: torch.from_numpy(a).cuda()) if device else (lambda a: a)
    got.partition_batch(rb, cb, *[[put(a) for a in p] for p in (us, is_, xs)])
    want.partition_diag(rb, cb, u, i, np.concatenate(xs))
    for a, b in zip(got.block_stats(), want.block_stats()):
        assert np.array_equal(a, b)
    for ctx in (got, want):
        ctx.factor(3, warn=False)
    assert np.array_equal(got.predict(u, i), want.predict(u, i))


def test_what_is_refused():
    rb, cb, us, is_, xs = matrices([(8, 8, 20), (9, 5, 20)], 1)
    ctx = bs.Context()
    with pytest.raises(ValueError):
        ctx.partition_batch(rb, cb, us[:1], is_, xs)
    with pytest.raises(ValueError):
        ctx.partition_batch(rb, cb, us, [is_[0], is_[1][1:]], xs)
    bad = us[0].copy()
    bad[3] = 8                               # the other matrix's first row
    with pytest.raises(bs.BsvdError):
        ctx.partition_batch(rb, cb, [bad, us[1]], is_, xs)
    with pytest.raises(ValueError):
        serve.run_batch(ctx, [])
    ctx.partition_batch(rb, cb, us, is_, xs)
    assert ctx.nblocks == 2
