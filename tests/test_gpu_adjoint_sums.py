"""The gradient of the gains joins the FP32 sums of single rows in FP64."""
import numpy as np
import pytest

from paper_2306_15678_gb300 import configs
from paper_2306_15678_gb300.adjoint import AdjointMarch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [8, 64, 512, 2048])
def test_rows_of_a_pair_are_joined_in_fp64(n):
    """One step of the Kerr screen alone.  Rows are constant along x; even rows hold
    amplitude a, odd rows a / 4, and F - D is +-x on every other even row and y =
    2^-18 x on the odd ones.  dJ/dtheta_1 sums a_K u w |U|^2 (w = 4 (F - D) / sum D^2)
    over the points: the even rows' parts are +-A, equal in bits, and cancel; each
    odd row's is 2^-8 2^-18 A, below half a unit of A in FP32, so a pair joined in
    FP32 loses it whole.  Tolerance: the odd rows take up the transforms' rounding
    at the level of the even ones, 4 x 1e-6 relative, and the sum follows its fourth
    power."""
    cfg = configs.physics(n, 1.0, 0.5, configs.KERR)
    a2 = 1.0e12
    U = np.full((n, n), np.sqrt(a2), dtype=np.complex64)
    U[1::2] /= 4
    F = np.abs(U.astype(np.complex128)) ** 2
    x = 2.0 ** 24 * a2
    D = np.empty((n, n))
    D[0::4], D[2::4] = F[0::4] - x, F[2::4] + x
    D[1::2] = F[1::2] - 2.0 ** -18 * x
    fit = AdjointMarch(cfg, 1, 1, precision="fp32")
    fit.set_target(D)
    fit.forward(U)
    dth, _ = fit.backward()
    fit.close()
    k0 = 2 * np.pi * cfg["n0"] / cfg["lambda0"]
    u = np.abs(U[1, 0].astype(np.complex128)) ** 2
    w = 4 * 2.0 ** -18 * x / (D ** 2).sum()
    ref = (n * n // 2) * cfg["dz"] * k0 * cfg["n2"] * u * w * u
    assert abs(dth[1] / ref - 1) < 2e-5, (dth[1], ref)
