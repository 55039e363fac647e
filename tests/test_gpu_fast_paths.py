"""The branches that the sizes, intensities, launch shapes and pointers of a call
choose between, each at the edges where it takes over, against the same
operation in FP64 numpy or its other branch."""
import math

import numpy as np
import pytest
import torch

from paper_2306_15678_gb300 import beams, capi, configs
from paper_2306_15678_gb300.adjoint import AdjointMarch
from paper_2306_15678_gb300.grid import Grid

pytestmark = pytest.mark.gpu

IREF = 1.0e13


def pointwise_cfg(n, K, theta=configs.NOMINAL_THETA):
    """A step of the screen alone whose phase is u = I / 1e13 (Kerr) + 0.3 u^K
    and whose absorption number is about 0.1 u^(K-1)."""
    cfg = configs.physics(n, 1.0, 0.5, configs.KERR | configs.PLASMA | configs.MPA, theta)
    k0 = 2 * math.pi * cfg["n0"] / cfg["lambda0"]
    cfg.update(K=K, n2=1.0 / (cfg["dz"] * k0 * IREF), betaK=0.1 / (cfg["dz"] * max(K - 1, 1)) / IREF ** (K - 1))
    cfg["sigmaK"] = 0.3 * 2 / (k0 * cfg["dz"]) * cfg["rho_c"] / (cfg["rho_nt"] * cfg["tau_pl"]) / IREF ** K
    return cfg


def coefs(cfg):
    k0 = 2 * math.pi * cfg["n0"] / cfg["lambda0"]
    aK = cfg["dz"] * k0 * cfg["n2"] * IREF
    aP = -cfg["dz"] * k0 / 2 * cfg["sigmaK"] * cfg["rho_nt"] * cfg["tau_pl"] / cfg["rho_c"] * IREF ** cfg["K"]
    aA = -cfg["dz"] * cfg["betaK"] / 2 * IREF ** (cfg["K"] - 1)
    return aK, aP, aA


def screen_ref(U, cfg, exact):
    u = np.abs(U) ** 2 / IREF
    K, th = cfg["K"], cfg["theta"]
    aK, aP, aA = coefs(cfg)
    if not exact:
        return U * np.exp((th[1] - 1j * th[0]) * aK * u + (th[3] - 1j * th[2]) * aP * u ** K
                          + (th[4] + 1j * th[5]) * aA * u ** (K - 1))
    a = -2 * (K - 1) * aA * u ** (K - 1)
    l, km1 = np.log1p(a), K - 1.0
    with np.errstate(invalid="ignore", divide="ignore"):
        f1 = np.where(a == 0, 1.0, l / a if K == 2 else np.expm1((K - 2) / km1 * l) / (a * (K - 2) / km1))
        fk = np.where(a == 0, 1.0, -km1 * np.expm1(-l / km1) / a)
    return U * np.exp(-l / (2 * km1) - 1j * (aK * u * f1 + aP * u ** K * fk))


def noise_field(n, umax, seed):
    """|U|^2 / 1e13 uniform in [0, umax), phases uniform."""
    rng = np.random.default_rng(seed)
    u = umax * rng.random((n, n))
    u[n // 2, n // 3] = 0.0
    return np.sqrt(u * IREF) * np.exp(2j * np.pi * rng.random((n, n)))


# largest u around which the short polynomials (phase 1/32), the middle ones (pi/4) and the
# series of the exact substep (a = 0.1 u^(K-1) <= 2^-7: u = 0.078 at K = 2, 0.69 at K = 8) hand over
@pytest.mark.parametrize("K,exact", [(8, False), (5, False), (8, True), (2, True), (5, True)])
@pytest.mark.parametrize("n", [8, 64, 512])
def test_screen_forms(n, K, exact):
    """FP32: the transforms around the screen leave at most 1e-6 relative (four
    transforms of log2 n stages at 2^-24 per stage and part, added in squares); the
    screen's phase a_K u + a_P u^K follows the relative error of u (2^-22: its parts,
    their squares, the sum and the scale) once in the first term and K times in the
    second.  FP64: the same with 1e-13 and 2^-51."""
    for umax in (0.02, 0.0312, 0.0625, 0.3, 0.69, 0.79, 4.0):
        if K == 8 and umax > 2:
            umax = 1.5
        cfg = dict(pointwise_cfg(n, K), screen="exact" if exact else "frozen")
        U = noise_field(n, umax, 7)
        for prec, ct in (("fp32", np.complex64), ("fp64", np.complex128)):
            V = U.astype(ct)
            ref = screen_ref(V.astype(np.complex128), cfg, exact)
            with Grid(cfg, precision=prec) as g:
                got = g.load(V).step(1).field()
            aK, aP, _ = coefs(cfg)
            base, eps = (1e-13, 2.0 ** -51) if prec == "fp64" else (1e-6, 2.0 ** -22)
            tol = base + (abs(aK) * umax + K * abs(aP) * umax ** K) * eps
            err = np.linalg.norm(got - ref) / np.linalg.norm(ref)
            assert err < tol, (umax, prec, err, tol)


@pytest.mark.parametrize("n", [8, 64, 512, 1024])
def test_adjoint_stash_orders(n):
    """The re-march leaves the fields in the order of its row pass's threads: natural
    for radix 8, permuted for radix 16 from 512 points on.  Both give the gradients
    of the FP64 adjoint to the scope's 1e-3 (a wrong order is an O(1) error)."""
    cfg = configs.physics(n, 8.0, 1.0, configs.ALL_TERMS, (1.1, 0.02, 1.0, 0.0, 1.0, 0.0))
    beam = dict(w0=1.0, P=50.0 * configs.critical_power(), amp=0.05, ell_cells=2.0, phase=0.1)
    U = beams.make_field(dict(cfg, beam=dict(beam, seed=3, phase_seed=4)))
    D = np.abs(beams.make_field(dict(cfg, beam=dict(beam, w0=1.1, seed=5, phase_seed=6)))) ** 2
    got = []
    for prec, launch in (("fp64", None), ("fp32", {"cols": 1, "row_radix": 16}),
                         ("fp32", {"cols": capi.NLSE_COL_R8 | 1, "row_radix": 8})):
        fit = AdjointMarch(cfg, 5, 2, precision=prec)
        if launch:
            fit.set_launch(launch)
        fit.set_target(D)
        loss = fit.forward(U)
        dth, dU = fit.backward()
        got.append((loss, dth, dU.cpu().numpy().astype(np.complex128)))
        fit.close()
    ref = got[0]
    for loss, dth, dU in got[1:]:
        assert abs(loss / ref[0] - 1) < 1e-3
        assert np.linalg.norm(dth - ref[1]) < 1e-3 * np.linalg.norm(ref[1])
        assert np.linalg.norm(dU - ref[2]) < 1e-3 * np.linalg.norm(ref[2])


@pytest.mark.parametrize("n,conn", [(8, 4), (16, 8), (64, 8), (256, 4)])
def test_hot_area_labels_at_any_alignment(n, conn):
    """Device labels that the 16-byte accesses cannot use give the same labels."""
    cfg = configs.physics(n, 1.0, 0.5, configs.KERR)
    with Grid(cfg, precision="fp32") as g:
        g.load(noise_field(n, 1.0, n).astype(np.complex64))
        count, ref = g.hot_areas(0.55 * IREF, conn, labels=True)
        buf = torch.full((n * n + 8,), -7, dtype=torch.int32, device="cuda")
        for off in (0, 1, 2, 3):
            buf.fill_(-7)
            assert capi.nlse_hot_areas(g.h, 0.55 * IREF, conn, buf.data_ptr() + 4 * off, True) == count
            out = buf.cpu().numpy()
            assert np.array_equal(out[off:off + n * n].reshape(n, n), ref)
            assert (out[:off] == -7).all() and (out[off + n * n:] == -7).all()


@pytest.mark.parametrize("prec,tol", [("fp64", 1e-12), ("fp32", 1e-4)])
@pytest.mark.parametrize("n", [8, 64, 512, 2048])
def test_moment_powers(n, prec, tol):
    """Every kind of exponent (0, 1, 2, odd, even, the largest); positive terms, so the
    sums follow the relative error of I^p: 16 times 2^-53 and the transforms', or
    16 times the FP32 load and readout's 1e-6."""
    L = 0.02 * n
    cfg = configs.physics(n, L, 0.5, configs.KERR)
    u = 0.5 + 0.5 * np.random.default_rng(n).random((n, n))
    U = np.sqrt(u).astype(np.complex64).astype(np.complex128)
    x = (np.arange(n) - n / 2 + 0.5) * (L / n)
    r2 = x[:, None] ** 2 + x[None, :] ** 2
    pq = [(1, 0), (1, 1), (2, 2), (3, 5), (4, 0), (7, 3), (16, 16), (6, 12)]
    with Grid(cfg, precision=prec) as g:
        got = g.load(U if prec == "fp64" else U.astype(np.complex64)).moments(pq)
    for k, (p, q) in enumerate(pq):
        ref = float((np.abs(U) ** (2 * p) * r2 ** q).sum()) * (L / n) ** 2
        assert abs(got[k] / ref - 1) < tol, (p, q, got[k] / ref - 1)
