"""The Rayleigh-Ritz solve (Cholesky QR, Jacobi, the convergence test) on
blocks whose shorter side is around its widths: odd and even sizes, one
column, fewer columns than the subspace and just more, against numpy's SVD
of the centred block in float64."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402


@pytest.mark.parametrize("k", [4, 20, 40])          # subspaces of 16, 32, 64
@pytest.mark.parametrize("s", [1, 2, 3, 7, 15, 16, 17, 30, 31, 32, 33, 47, 63,
                               64, 65, 129])
def test_singular_values_at_the_subspace_widths(s, k):
    m = 211
    r = synth.random_ratings(70 + s, m, s, max(1, int(0.6 * m * s)), 0)
    part = oracle.partition(m, s, r.u_train, r.i_train, r.x_train, 1, 1)
    sv = np.linalg.svd(oracle.dense_block(part, 0), compute_uv=False)
    with bs.Context() as ctx:
        ctx.partition(m, s, r.u_train, r.i_train, r.x_train, 1, 1)
        assert ctx.factor(k, warn=False) == bs.OK
        g = ctx.get_block(0)
    ke = min(k, s)
    assert g["keff"] == ke
    # the solver's residual bar is 1e-5 theta_1 (theta = sigma^2)
    assert np.all(np.abs(g["sigma"] - sv[:ke]) <= 1e-5 * sv[0])
    live = g["sigma"] > 1e-3 * sv[0]
    V = g["V"][:, live].astype(np.float64)
    assert np.max(np.abs(V.T @ V - np.eye(live.sum()))) <= 2e-4


def test_dependent_columns_are_refilled():
    """Identical columns: the basis collapses and columns are refilled."""
    m, n = 150, 90
    u, i = np.divmod(np.arange(m * n), n)
    x = (1 + (u * 7) % 5).astype(np.float32)
    with bs.Context() as ctx:
        ctx.partition(m, n, u.astype(np.int32), i.astype(np.int32), x, 1, 1)
        ctx.factor(10, warn=False)
        s = ctx.get_block(0)["sigma"]
    want = np.linalg.svd((x - x.mean()).reshape(m, n).astype(np.float64),
                         compute_uv=False)
    assert abs(s[0] - want[0]) <= 1e-5 * want[0]
    assert np.all(s[1:] <= 2e-3 * want[0])
