"""Masks with a region at almost every pixel: the labelling and the lens list at the
edges of the strips that a warp takes (32 pixels up to n = 512, 128 beyond), where
the answer is known without a flood fill."""
import numpy as np
import pytest

from paper_2306_15678_gb300 import configs
from paper_2306_15678_gb300.grid import Grid

pytestmark = pytest.mark.gpu


def patterns(n):
    """name -> (mask, labels with 4 neighbours, labels with 8)"""
    y, x = np.mgrid[:n, :n]
    own = (y * n + x).astype(np.int32)
    board = (x + y) % 2 == 0
    yield "board", board, np.where(board, own, -1), np.where(board, 0, -1)
    dots = (x % 2 == 0) & (y % 2 == 0)
    yield "dots", dots, np.where(dots, own, -1), np.where(dots, own, -1)
    cols = x % 2 == 1
    yield "columns", cols, np.where(cols, x, -1), np.where(cols, x, -1)
    # rising diagonals, three apart: 8 neighbours join each to its top right end
    diag = (x + y) % 3 == 0
    s = x + y
    top = np.where(s < n, s, (s - n + 1) * n + n - 1)
    yield "diagonals", diag, np.where(diag, own, -1), np.where(diag, top, -1)


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("n", [8, 16, 32, 512, 1024, 2048])
def test_labels_and_lens_centres(n, prec):
    cfg = configs.physics(n, 0.005 * n, 0.5, configs.KERR | configs.DIFFRACTION)
    lens = dict(l_dif=1e-30, w_l=1e12, re=[], im=[])
    with Grid(cfg, precision=prec) as g:
        for name, mask, lab4, lab8 in patterns(n):
            U = np.sqrt(np.where(mask, 2e12, 1e11)).astype(g.cdtype)
            for conn, want in ((4, lab4), (8, lab8)):
                g.load(U)
                roots = np.unique(want[want >= 0])
                count, labels = g.hot_areas(1e12, conn, labels=True)
                assert count == len(roots), (name, conn)
                assert np.array_equal(labels, want), (name, conn)
                # a lens's centre is its first pixel of the largest w_dif: with equal
                # pixels up to rounding, any pixel of the region; one per region
                k, cent, _ = g.effective_lens(dict(lens, conn=conn))
                assert k == len(roots) and np.all(np.diff(cent) > 0), (name, conn)
                assert np.array_equal(np.sort(want.ravel()[cent]), roots), (name, conn)
