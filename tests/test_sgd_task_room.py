"""Room for the blocked SGD's tasks when some ratings have ids out of range:
they are sorted as cell (0, 0) of block 0, which an empty first block does not
have. The bound against the tasks of a model of the order, on the CPU; then
the call itself."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
import synth
from oracle import sgd as osgd

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1907_07410_gb300", "csrc")


@pytest.fixture(scope="module")
def max_tasks(tmp_path_factory):
    d = tmp_path_factory.mktemp("tasks")
    src, lib = str(d / "t.cpp"), str(d / "t.so")
    with open(src, "w") as f:
        f.write('#include "sgd_tasks.h"\n'
                'extern "C" long long max_tasks(long long nnz, int diag, int '
                'own, long long p, long long q, long long m, long long n) {\n'
                '  return bsvd::sgd_max_tasks(nnz, diag, own, p, q, m, n);\n}\n')
    subprocess.check_call(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                           "-o", lib, src])
    f = ctypes.CDLL(lib).max_tasks
    f.restype = ctypes.c_longlong
    f.argtypes = [ctypes.c_longlong, ctypes.c_int, ctypes.c_int] + \
        [ctypes.c_longlong] * 4
    return f


def tasks(rb, cb, u, i, diag):
    """Distinct (step, owner's local index, block in the step) of the ratings,
    (0, 0, 0) for the bad ones."""
    p, q, m, n = len(rb) - 1, len(cb) - 1, rb[-1], cb[-1]
    own = n <= m
    seen = set()
    for a, b in zip(u, i):
        key = (0, 0, 0)
        if 0 <= a < m and 0 <= b < n:
            bi = int(np.searchsorted(rb, a, side="right")) - 1
            bj = int(np.searchsorted(cb, b, side="right")) - 1
            lo = b - cb[bj] if own else a - rb[bi]
            if diag:
                key = (0, lo, bi) if bi == bj else key
            elif p >= q:
                key = ((bi - bj) % p, lo, bj)
            else:
                key = ((bj - bi) % q, lo, bi)
        seen.add(key)
    return len(seen)


def bounds(rng, size, parts):
    """Non-decreasing bounds, empty blocks among them."""
    b = np.sort(rng.integers(0, size + 1, parts - 1))
    if rng.random() < 0.5:
        b[:rng.integers(0, parts)] = 0
    return np.concatenate([[0], b, [size]])


def example(empty_rows=False):
    """Every cell rated, the first block empty on the owner's side, one id out
    of range in place of a rating of a cell that has others of its owner."""
    m, n = (127, 200) if empty_rows else (200, 127)
    u, i = np.divmod(np.arange(m * n), n)
    u[500] = m
    rb = np.array([0, 0, m] if empty_rows else [0, m])
    cb = np.array([0, n] if empty_rows else [0, 0, n])
    return m, n, rb, cb, u.astype(np.int32), i.astype(np.int32)


@pytest.mark.parametrize("empty_rows", [False, True])
def test_room_for_an_empty_first_block(max_tasks, empty_rows):
    m, n, rb, cb, u, i = example(empty_rows)
    p, q = len(rb) - 1, len(cb) - 1
    need = tasks(rb, cb, u, i, False)
    assert need == 128
    assert max_tasks(len(u), 0, n <= m, p, q, m, n) >= need


def test_room_for_random_grids(max_tasks):
    rng = np.random.default_rng(3)
    for _ in range(400):
        diag = bool(rng.integers(0, 2))
        m, n = (int(v) for v in rng.integers(1, 12, 2))
        p = int(rng.integers(1, 5))
        q = p if diag else int(rng.integers(1, 5))
        rb, cb = bounds(rng, m, p), bounds(rng, n, q)
        u, i = (a.ravel() for a in np.meshgrid(np.arange(-1, m + 1),
                                               np.arange(-1, n + 1)))
        assert max_tasks(len(u), diag, n <= m, p, q, m, n) >= \
            tasks(rb, cb, u, i, diag)


@pytest.mark.gpu
@pytest.mark.parametrize("empty_rows", [False, True])
def test_bad_id_beside_an_empty_first_block(empty_rows):
    """The call is refused, and the context goes on as if it had not been."""
    bs = pytest.importorskip("paper_1907_07410_gb300")
    m, n, rb, cb, u, i = example(empty_rows)
    x = (1 + np.arange(len(u)) % 5).astype(np.float32)
    good = u < m
    with bs.Context() as ctx:
        ctx.partition(m, n, u[good], i[good], x[good], len(rb) - 1,
                      len(cb) - 1, row_bounds=rb, col_bounds=cb)
        with pytest.raises(bs.BsvdError):
            ctx.sgd_prepare(u, i, x)
        ctx.sgd_prepare(u[good], i[good], x[good])
        P0, Q0 = synth.sgd_start(m, n, 4, 5)
        ctx.sgd_train(P0, Q0, max_steps=1, delta=-1e300)
        got = ctx.sgd_get()
    ref = osgd.train(oracle.make_grid(m, n, len(rb) - 1, len(cb) - 1,
                                      row_bounds=rb, col_bounds=cb),
                     u[good], i[good], x[good], P0, Q0, 1, delta=-1e300)
    for a, b in zip(got, (ref.P, ref.Q, ref.bu, ref.bi)):
        assert np.array_equal(a, b)
