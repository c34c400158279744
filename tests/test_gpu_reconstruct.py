"""The dense reconstruction against mu + P V^T in float64 from the block's own
factors, element by element, at the edges of its tiles and of the rule that
groups rows by where they start in a 128-byte line."""
import numpy as np
import pytest

import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import paper_1907_07410_gb300 as bs  # noqa: E402

# three tf32 products: the dropped terms are below 2^-21 of sum |p||v|, and
# each of the at most 3 * 56 additions rounds by at most 2^-23 of it
REL = 2.0 ** -21 + 168 * 2.0 ** -23


def check(m, n, k, offset=0, add_mean=True, density=0.2):
    r = synth.random_ratings(50 + m + n, m, n, max(1, int(m * n * density)), 0)
    with bs.Context() as ctx:
        ctx.partition(m, n, r.u_train, r.i_train, r.x_train, 1, 1)
        ctx.factor(k, warn=False)
        g = ctx.get_block(0)
        buf = torch.full((offset + m * n + 64,), -77.0, device="cuda")
        ctx.reconstruct(0, add_mean=add_mean, out=buf[offset:])
        got = buf.cpu().numpy()
    P, V = g["P"].astype(np.float64), g["V"].astype(np.float64)
    want = P @ V.T + (g["mu"] if add_mean else 0.0)
    # F_s times sigma is rounded once more on its way to P or V
    scale = np.abs(P) @ np.abs(V).T + (abs(g["mu"]) if add_mean else 0.0)
    out = got[offset:offset + m * n].reshape(m, n)
    assert np.all(np.abs(out - want) <= (REL + 2.0 ** -22) * scale + 1e-30)
    # nothing beside the block is written
    assert np.all(got[:offset] == -77.0)
    assert np.all(got[offset + m * n:] == -77.0)


@pytest.mark.parametrize("m,n", [(1, 1), (1, 200), (200, 1), (127, 127),
                                 (128, 128), (129, 129), (128, 31), (33, 160),
                                 (257, 130), (300, 96), (640, 97)])
@pytest.mark.parametrize("offset", [0, 1])
def test_tile_edges(m, n, offset):
    check(m, n, 7, offset, add_mean=offset == 0)


# 512 rows of one residue and more: G = 32, 16, 8, 1 and 2 residues, the last
# row of each short of, at and past a tile
@pytest.mark.parametrize("m,n,offset", [(16384, 33, 0), (16387, 35, 3),
                                        (16415, 129, 2), (8200, 34, 1),
                                        (4100, 36, 0), (1000, 64, 0),
                                        (1000, 64, 5), (1030, 48, 7)])
def test_rows_grouped_by_residue(m, n, offset):
    check(m, n, 5, offset, density=0.1)


@pytest.mark.parametrize("k", [1, 8, 9, 32, 33, 40, 56])
def test_ranks_across_the_operand_atoms(k):
    check(300, 211, k, 1)
