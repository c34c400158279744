"""The blocked SGD's waits end. A task list made by hand waits for versions of
the parameters that no rating leaves, with a short limit: every warp leaves,
the error word says that a wait gave up, and the next training on the same GPU
is the oracle's to the bit."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle
import synth
from oracle import sgd as osgd

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402
from paper_1907_07410_gb300 import build  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))
TIMEOUT = 16                # kErrTimeout
POLLS = 1 << 13


@pytest.fixture(scope="module")
def give_up(tmp_path_factory):
    lib = str(tmp_path_factory.mktemp("sgd") / "give_up.so")
    subprocess.check_call(
        [build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", lib,
         os.path.join(HERE, "sgd_give_up.cu"), build.build(),
         "-Xlinker", "-rpath," + os.path.dirname(build.LIB)])
    f = ctypes.CDLL(lib).give_up
    f.argtypes = [ctypes.c_int] * 4 + [ctypes.c_uint] * 3 + [ctypes.c_void_p]

    def run(*args):
        out = (ctypes.c_ulonglong * 4)()
        assert f(*args, out) == 0
        return list(out)
    return run


# k: each lane layout (both sides in half a warp, a lane each, every lane a
# bias); tasks: one warp's, and more than the resident warps'
@pytest.mark.parametrize("tasks", [2, 9, 4000])
@pytest.mark.parametrize("k", [3, 20, 32])
@pytest.mark.parametrize("f32", [0, 1])
def test_a_version_that_never_comes(give_up, f32, k, tasks):
    for other, own in ((1 << 20, 0), (0, 1 << 20)):
        # users = tasks: with nothing to wait for, no wait gives up
        err, claimed, _, stop = give_up(f32, k, tasks, tasks, 0, 0, POLLS)
        assert (err, stop) == (0, 0) and claimed >= tasks
        err, claimed, _, stop = give_up(f32, k, tasks, tasks, other, own, POLLS)
        assert (err, stop) == (TIMEOUT, 1) and claimed >= 2
    r = synth.random_ratings(43, 60, 40, 900, 0)
    P0, Q0 = synth.sgd_start(60, 40, k, 3)
    with bs.Context() as ctx:
        ctx.partition(60, 40, r.u_train, r.i_train, r.x_train, 3, 2)
        ctx.sgd_prepare(r.u_train, r.i_train, r.x_train)
        ctx.sgd_train(P0, Q0, max_steps=1, delta=-1e300,
                      precision=bs.SGD_FP32 if f32 else bs.SGD_FP64)
        got = ctx.sgd_get()
    ref = osgd.train(oracle.make_grid(60, 40, 3, 2), r.u_train, r.i_train,
                     r.x_train, P0, Q0, 1, delta=-1e300,
                     dtype=np.float32 if f32 else np.float64)
    for a, b in zip(got, (ref.P, ref.Q, ref.bu, ref.bi)):
        assert np.array_equal(a, b)
