"""Ids that one matrix of a batch does not have. Both of a rating's ids out of
range by the next matrix's offsets make a cell of that matrix in the stacked
coordinates, so the block diagonal alone does not show them."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402
from paper_1907_07410_gb300 import serve  # noqa: E402

SIZES = [(8, 8), (9, 5), (6, 7)]


def batch(seed=1):
    rng = np.random.default_rng(seed)
    us, is_, xs = [], [], []
    for m, n in SIZES:
        cells = rng.permutation(m * n)[:20]
        us.append((cells // n).astype(np.int32))
        is_.append((cells % n).astype(np.int32))
        xs.append(rng.integers(1, 6, 20).astype(np.float32))
    rb, cb = ([0] + list(np.cumsum([s[d] for s in SIZES])) for d in (0, 1))
    return rb, cb, us, is_, xs


@pytest.mark.parametrize("b,u,i", [
    (0, 8, 8),                  # matrix 1's first cell
    (1, -1, -1),                # matrix 0's last cell
    (1, 9 + 5, 5 + 6),          # matrix 2's last cell
    (2, -17, -13),              # matrix 0's first cell
    (2, 6, 7), (0, -1, -1),     # outside the batch
    (0, 2**31 - 1, 2**31 - 1), (2, -2**31, -2**31),
])
def test_a_rating_of_another_matrix(b, u, i):
    rb, cb, us, is_, xs = batch()
    ctx = bs.Context()
    us[b][3], is_[b][3] = u, i
    with pytest.raises(bs.BsvdError):
        ctx.partition_batch(rb, cb, us, is_, xs)


@pytest.mark.parametrize("which", [0, 1, 2])
def test_lengths_that_cancel_over_the_batch(which):
    """One array of each kind a matrix, all three of a matrix equally long:
    here one rating of matrix 0's moves to matrix 1 in one of the three."""
    rb, cb, us, is_, xs = batch()
    a = (us, is_, xs)[which]
    a[0], a[1] = a[0][:-1], np.concatenate([a[0][-1:], a[1]])
    with pytest.raises((bs.BsvdError, ValueError)):
        bs.Context().partition_batch(rb, cb, us, is_, xs)
    reqs = [serve.Request(m, n, 2, u, i, x, u[:1], i[:1])
            for (m, n), u, i, x in zip(SIZES, us, is_, xs)]
    with pytest.raises((bs.BsvdError, ValueError)):
        serve.run_batch(bs.Context(), reqs)


def requests(b=None, qr=None, qc=None):
    _, _, us, is_, xs = batch()
    reqs = [serve.Request(m, n, 2, u, i, x, u[:3], i[:3])
            for (m, n), u, i, x in zip(SIZES, us, is_, xs)]
    if b is not None:
        reqs[b].qr = np.array([0, qr], np.int32)
        reqs[b].qc = np.array([0, qc], np.int32)
    return reqs


@pytest.mark.parametrize("b,qr,qc", [(0, 8, 8), (1, -1, -1), (1, 14, 11),
                                     (2, -17, -13), (0, 8, 0), (1, 0, -1)])
def test_a_prediction_of_another_request(b, qr, qc):
    """A cell of another request's matrix is no answer to this one's query."""
    with bs.Context() as ctx:
        with pytest.raises(bs.BsvdError):
            serve.run_batch(ctx, requests(b, qr, qc))
        got = serve.run_batch(ctx, requests())
    assert [len(y) for y in got] == [3, 3, 3]


def test_requests_of_two_dimensions():
    """Columns of ids are stacked by the host: the same ids, the same checks."""
    def columns(reqs):
        for q in reqs:
            q.r, q.c, q.x = (a.reshape(-1, 1) for a in (q.r, q.c, q.x))
        return reqs
    with bs.Context() as ctx:
        for a, b in zip(serve.run_batch(ctx, columns(requests())),
                        serve.run_batch(ctx, requests())):
            assert np.array_equal(a, b)
        bad = requests()
        bad[0].r[3], bad[0].c[3] = 8, 8
        with pytest.raises(bs.BsvdError):
            serve.run_batch(ctx, columns(bad))


def test_queries_whose_lengths_cancel():
    reqs = requests()
    reqs[0].qr, reqs[1].qc = reqs[0].qr[:2], reqs[1].qc[:2]
    with bs.Context() as ctx:
        with pytest.raises((bs.BsvdError, ValueError)):
            serve.run_batch(ctx, reqs)
