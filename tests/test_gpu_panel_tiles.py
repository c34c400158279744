"""Panel products over more tiles than multiprocessors, with blocks that stop
at different steps (a third of them hold no rating and stop at once): block
sides from less than one K stage to more than the stage ring, each subspace
width, against numpy's SVD of the centred blocks in float64."""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402


def ratings(s, p, density, seed):
    """Uniform ratings 1 .. 5; none in blocks (a, b) with (a + b) % 3 == 1."""
    rng = np.random.default_rng(seed)
    m = s * p
    u, i = np.divmod(rng.permutation(m * m)[: int(density * m * m)], m)
    keep = (u // s + i // s) % 3 != 1
    u, i = u[keep].astype(np.int32), i[keep].astype(np.int32)
    return u, i, rng.integers(1, 6, len(u)).astype(np.float32)


@pytest.mark.parametrize("k", [4, 20, 40])          # subspaces of 16, 32, 64
@pytest.mark.parametrize("s,p", [(31, 14), (65, 13), (129, 9), (300, 7),
                                 (577, 3)])
def test_tiles_of_running_and_stopped_blocks(s, p, k):
    m = n = s * p
    u, i, x = ratings(s, p, 0.2, 7 * s + k)
    part = oracle.partition(m, n, u, i, x, p, p)
    with bs.Context(profile=1, loop=1) as ctx:
        ctx.partition(m, n, u, i, x, p, p)
        assert ctx.factor(k, warn=False) == bs.OK
        ph = ctx.phase_times()
        assert 0 < ph["eigen_filter"] <= ph["eigen"]
        for b in sorted({0, 1, p + 1, p * p // 2, p * p - 1}):
            g = ctx.get_block(b)
            sv = np.linalg.svd(oracle.dense_block(part, b), compute_uv=False)
            ke = min(k, s)
            # the solver's residual bar is 1e-5 theta_1 (theta = sigma^2)
            assert np.all(np.abs(g["sigma"] - sv[:ke]) <= 1e-5 * sv[0])
