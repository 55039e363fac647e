"""The FP32 adjoint under launch shapes that are all named, so that a change of a
default cannot make two arms of a comparison the same."""
import numpy as np
import pytest

from paper_2306_15678_gb300 import beams, capi, configs
from paper_2306_15678_gb300.adjoint import AdjointMarch

pytestmark = pytest.mark.gpu

TMA, R8, STAGED = capi.NLSE_COL_TMA, capi.NLSE_COL_R8, capi.NLSE_ROW_STAGED


def gradient(n, steps, ckpt, cols, row_radix):
    cfg = configs.scaled(configs.cfg_dense_fp32(), n)
    U0 = beams.make_field(cfg).astype(np.complex64)
    D = np.abs(beams.make_field(dict(cfg, beam=dict(cfg["beam"], w0=1.05, seed=7)))) ** 2
    fit = AdjointMarch(cfg, steps, ckpt, precision="fp32")
    fit.set_launch({"cols": cols, "row_radix": row_radix})
    fit.set_target(D)
    loss = fit.forward(U0)
    dth, dU = fit.backward()
    fit.close()
    return loss, dth, dU.cpu().numpy()


def test_column_tiles_and_row_staging_keep_the_bits():
    """Single staged columns, interleaved pairs and two pairs, per-thread tiles, and
    both radix-16 row passes, with the conjugated tables of the backward sweep."""
    ref = gradient(2048, 4, 2, TMA | 1, 16)
    for cols, rows in ((TMA | 2, 16), (TMA | 4, 16), (2, 16), (TMA | 1, STAGED | 16)):
        got = gradient(2048, 4, 2, cols, rows)
        assert got[0] == ref[0], (cols, rows)
        assert np.array_equal(got[1], ref[1]) and np.array_equal(got[2], ref[2]), (cols, rows)


@pytest.mark.parametrize("n", [2048, 4096, 8192])
def test_stash_orders_of_the_large_grids(n):
    """Natural stash order (radix 8) against the permuted one (radix 16, which at 8192
    has a formula of its own): the same gradients to the 1e-3 of FP32 gradients (a wrong
    order is an O(1) error)."""
    a = gradient(n, 2, 2, TMA | 1, 16)
    b = gradient(n, 2, 2, R8 | 1, 8)
    assert abs(a[0] / b[0] - 1) < 1e-4
    assert np.linalg.norm(a[1] - b[1]) < 1e-3 * np.linalg.norm(b[1])
    assert np.linalg.norm(a[2] - b[2]) < 1e-3 * np.linalg.norm(b[2])
