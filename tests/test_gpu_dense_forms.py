"""What the partition keeps of the dense blocks: the exact Gram's planes alone
(from which the cells are rebuilt) when every rating is a small whole or half
offset from its block's rounded mean, else the float32 cells. Counts, means
and cells are compared with the oracle's bit for bit."""
import numpy as np
import pytest

import oracle
import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402


def check_partition(ctx, part, nb):
    cnt, mu = ctx.block_stats()
    assert np.array_equal(cnt, part.counts)
    assert np.array_equal(mu, part.mu32)
    for b in range(nb):
        got = ctx.get_block(b, want_factors=False, want_dense=True)["dense"]
        assert np.array_equal(got, oracle.dense_block(part, b, fp32=True)), b


def check_sigma(ctx, part, k, nb):
    for b in range(nb):
        B = oracle.dense_block(part, b)
        sv = np.linalg.svd(B, compute_uv=False)[:k]
        s = ctx.get_block(b)["sigma"]
        assert np.all(np.abs(s - sv[:len(s)]) <= 1e-5 * sv[0]), b


def ratings(scale, seed=80, m=230, n=170, nnz=9000):
    r = synth.random_ratings(seed, m, n, nnz, 0)
    rng = np.random.default_rng(seed)
    u, i = r.u_train, r.i_train
    x = {"stars": lambda: rng.integers(1, 6, nnz),
         "halves": lambda: rng.integers(1, 11, nnz) / 2,
         "quarters": lambda: rng.integers(4, 21, nnz) / 4,
         "wide": lambda: rng.integers(-200, 201, nnz),
         "wide halves": lambda: rng.integers(-250, 251, nnz) / 2,
         "tiny": lambda: np.where(np.arange(nnz) == 77, 1e-9,
                                  rng.integers(1, 6, nnz))}[scale]()
    return m, n, u, i, x.astype(np.float32)


@pytest.mark.parametrize("scale,path", [("stars", 2), ("halves", 2),
                                        ("quarters", 1), ("wide", 2),
                                        ("wide halves", 2), ("tiny", 2)])
@pytest.mark.parametrize("panel", [0, 1])
def test_forms_of_float32_blocks(scale, path, panel):
    m, n, u, i, x = ratings(scale)
    part = oracle.partition(m, n, u, i, x, 2, 3)
    with bs.Context(panel_path=panel) as ctx:
        ctx.partition(m, n, u, i, x, 2, 3)
        check_partition(ctx, part, 6)
        assert ctx.factor(6) == bs.OK
        assert ctx.gram_path() == path
        check_sigma(ctx, part, 6, 6)


def test_forced_tensor_gram_takes_whole_ratings_only():
    m, n, u, i, x = ratings("halves")
    with bs.Context(gram_path=2) as ctx:
        ctx.partition(m, n, u, i, x, 2, 3)
        with pytest.raises(bs.BsvdError) as e:
            ctx.factor(6)
        assert e.value.status == bs.EINVAL
        x = np.ceil(x)
        ctx.partition(m, n, u, i, x, 2, 3)
        assert ctx.factor(6) == bs.OK and ctx.gram_path() == 2


def test_one_context_through_every_form():
    """The cells' storage of one partition is not the next one's."""
    with bs.Context() as ctx:
        for scale in ("stars", "quarters", "halves", "tiny", "stars"):
            m, n, u, i, x = ratings(scale, seed=81)
            part = oracle.partition(m, n, u, i, x, 3, 2)
            ctx.partition(m, n, u, i, x, 3, 2)
            check_partition(ctx, part, 6)
            for _ in range(2):                # the host's loop, the graph
                assert ctx.factor(5) == bs.OK
                check_sigma(ctx, part, 5, 6)


@pytest.mark.parametrize("precision", ["BF16", "TF32"])
def test_other_forms_keep_their_blocks(precision):
    m, n, u, i, x = ratings("halves", seed=82)
    part = oracle.partition(m, n, u, i, x, 2, 2)
    with bs.Context(precision=getattr(bs, precision)) as ctx:
        ctx.partition(m, n, u, i, x, 2, 2)
        cnt, mu = ctx.block_stats()
        assert np.array_equal(mu, part.mu32)
        for b in range(4):
            got = ctx.get_block(b, want_factors=False, want_dense=True)["dense"]
            want = oracle.dense_block(part, b, fp32=True).astype(np.float32)
            if precision == "BF16":
                want = torch.from_numpy(want).bfloat16().float().numpy()
            assert np.array_equal(got, want)


# in order of blocks (a warp's ratings share one) and shuffled; with low words
# that carry; tables that fit and do not
@pytest.mark.parametrize("order", ["blocks", "shuffled"])
@pytest.mark.parametrize("p,q", [(1, 1), (4, 4), (32, 16), (513, 1), (60, 40)])
def test_exact_sums_of_fractional_ratings(order, p, q):
    m, n, nnz = 1100, 700, 20000
    r = synth.random_ratings(83, m, n, nnz, 0)
    rng = np.random.default_rng(84)
    x = (rng.uniform(-5, 5, nnz) + rng.integers(0, 2, nnz) * 0.37
         ).astype(np.float32)
    x[::3] = np.round(x[::3])
    x[np.abs(x) < 0.01] = 0.5         # sums are exact from 2^-9 on
    part = oracle.partition(m, n, r.u_train, r.i_train, x, p, q)
    key = (r.u_train // -(-m // p)) * q + r.i_train // -(-n // q)
    o = np.argsort(key, kind="stable") if order == "blocks" else \
        rng.permutation(nnz)
    with bs.Context() as ctx:
        ctx.partition(m, n, r.u_train[o], r.i_train[o], x[o], p, q)
        cnt, mu = ctx.block_stats()
    assert np.array_equal(cnt, part.counts)
    assert np.array_equal(mu, part.mu32)
