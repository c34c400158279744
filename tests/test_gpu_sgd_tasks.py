"""The blocked SGD's tasks (one owner's ratings in one block, run by a warp
while other warps run other tasks) against the sequential oracle, at the
sizes where the order or the lane layout can go wrong. Both sides round every
operation once and process every user's and every item's ratings in the same
order, so the bar is bit equality."""
import numpy as np
import pytest

import oracle
import synth
from oracle import sgd as osgd

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402


def check(m, n, u, i, x, p, q, k, f32, steps=2, grid_kw=None, owned=None):
    P0, Q0 = synth.sgd_start(m, n, k, 29)
    u, i = np.asarray(u, np.int32), np.asarray(i, np.int32)
    x = np.asarray(x, np.float32)
    with bs.Context() as ctx:
        if owned is not None:
            ctx.set_owned(owned)
        ctx.partition(m, n, u, i, x, p, q, **(grid_kw or {}))
        ctx.sgd_prepare(u, i, x)
        hist, ran = ctx.sgd_train(P0, Q0, max_steps=steps, delta=-1e300,
                                  precision=bs.SGD_FP32 if f32
                                  else bs.SGD_FP64)
        got = ctx.sgd_get()
    ref = osgd.train(oracle.make_grid(m, n, p, q, **(grid_kw or {})), u, i, x,
                     P0, Q0, steps, delta=-1e300,
                     dtype=np.float32 if f32 else np.float64)
    assert ran == ref.steps_run == steps
    for a, b in zip(got, (ref.P, ref.Q, ref.bu, ref.bi)):
        assert np.array_equal(a, b)
    np.testing.assert_allclose(hist, ref.rmse, rtol=1e-12, atol=0)


# lanes: both sides in half a warp up to 15 factors, a lane each up to 31,
# every lane a bias at 32
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("k", [1, 2, 14, 15, 16, 17, 30, 31, 32])
def test_ranks_on_both_lane_layouts(k, f32):
    r = synth.random_ratings(41, 90, 70, 2500, 0)
    check(90, 70, r.u_train, r.i_train, r.x_train, 3, 2, k, f32)


# users own the tasks when there are fewer of them than items
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("m,n,p,q", [(60, 200, 2, 5), (200, 60, 5, 2),
                                     (1, 150, 1, 3), (150, 1, 3, 1),
                                     (64, 64, 64, 64), (33, 257, 7, 3)])
def test_either_side_owns(m, n, p, q, f32):
    r = synth.random_ratings(42, m, n, min(3000, m * n // 2), 0)
    check(m, n, r.u_train, r.i_train, r.x_train, p, q, 6, f32)


# a task of exactly one, 31 .. 33 and 63 .. 65 ratings (32 are held at once)
@pytest.mark.parametrize("length", [1, 31, 32, 33, 63, 64, 65, 129])
def test_task_lengths_around_a_chunk(length):
    u = np.concatenate([np.arange(length), np.arange(length)[::3]])
    i = np.concatenate([np.zeros(length, int),
                        np.ones(len(np.arange(length)[::3]), int)])
    x = 1 + (np.arange(len(u)) * 7) % 5
    for f32 in (False, True):
        check(length, 2, u, i, x, 1, 1, 5, f32)


def test_repeated_cells_keep_input_order():
    rng = np.random.default_rng(6)
    u = rng.integers(0, 12, 900)
    i = rng.integers(0, 9, 900)
    x = rng.normal(3, 1, 900)
    for f32 in (False, True):
        check(12, 9, u, i, x, 3, 2, 7, f32)
        check(12, 9, np.full(200, 3), np.full(200, 4), x[:200], 3, 2, 7, f32)


def test_no_ratings():
    none = np.zeros(0, np.int32)
    with bs.Context() as ctx:
        ctx.partition(5, 4, none, none, none.astype(np.float32), 1, 1)
        ctx.sgd_prepare(none, none, none.astype(np.float32))
        P0, Q0 = synth.sgd_start(5, 4, 3, 1)
        ctx.sgd_train(P0, Q0, max_steps=2, delta=-1e300)
        P, Q, bu, bi = ctx.sgd_get()
    assert np.array_equal(P, P0) and np.array_equal(Q, Q0)
    assert not bu.any() and not bi.any()


def test_order_key_wider_than_64_bits():
    """Two sorts instead of one: 1024 x 512 blocks, one of them 2^23 - 1023
    users by 2^23 - 512 items (no block is held, so none is stored)."""
    m, n, p, q = 1 << 23, (1 << 23) - 1, 1024, 512
    rb = np.concatenate([[0], np.arange(m - p + 1, m + 1)]).astype(np.int64)
    cb = np.concatenate([[0], np.arange(n - q + 1, n + 1)]).astype(np.int64)
    rng = np.random.default_rng(8)
    u = np.concatenate([rng.integers(m - 40, m, 1200), rng.integers(0, m, 800)])
    i = np.concatenate([rng.integers(n - 30, n, 1200), rng.integers(0, n, 800)])
    check(m, n, u, i, rng.integers(1, 6, 2000), p, q, 1, True, steps=1,
          grid_kw=dict(row_bounds=rb, col_bounds=cb),
          owned=np.zeros(p * q, np.uint8))
