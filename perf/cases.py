"""What the framework is timed on: its public entry points (Grid, Batch,
AdjointMarch, NlseFluenceLoss) over the sizes, precisions and options that a
user of the march meets.

Every case starts from seeded beams of Eq. 7 made on the GPU (Gaussian beams
with correlated amplitude and phase noise, or a field of hot spots for the
diagnostics), in the physical regimes of ``configs``: sub-collapse powers and
step counts, so that rounding differences stay small and outputs can be
compared.  Every float that the framework hands out in 64 bits for an FP32 grid
(power, peak, moments, gradients of the gains) is returned as an FP32 value.

Kinds of case:
  march     load a device field, take `steps` z steps, read the field back
            (and the recorded power/peak history where diag_every > 0, or the
            downsampled fluence where ds > 0)
  batch     replay the captured graph of `steps` steps of many beams
  gradient  loss and gradients of the fluence-mismatch fit (checkpointed)
  plane     one plane: hot areas with labels, moments, then a turbulent layer and
            the effective-lens screen, and the field
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2306_15678_gb300 import configs
from paper_2306_15678_gb300.adjoint import AdjointMarch, NlseFluenceLoss
from paper_2306_15678_gb300.batch import Batch
from paper_2306_15678_gb300.grid import Grid

LENS = dict(l_dif=4e-4, w_l=1.0e11, conn=4,
            re=[(0.0313, 0.9, 40.0, 0.2), (0.0617, -0.5, 30.0, 1.0), (0.1037, 0.2, 20.0, -0.4)],
            im=[(0.0411, 0.3, 35.0, 0.1), (0.0807, 0.1, 15.0, 0.5)])  # no joint at a whole number of cells
GAINS = (1.1, 0.02, 1.0, 0.0, 1.0, 0.0)  # a gene of the fit: complex Kerr gain


def _march(name, n, precision, steps, L, w0, p_cr, dz, scheme="lie", screen="frozen", diag_every=0, ds=0):
    return dict(name=name, kind="march", n=n, precision=precision, steps=steps, L=L, w0=w0, p_cr=p_cr, dz=dz,
                scheme=scheme, screen=screen, diag_every=diag_every, ds=ds)


def listed():
    return [
        # the smallest call: one coarse test beam of the fit over a few steps; launches and host work are most of it
        _march("fit-beam-128", 128, "fp32", 6, 1.2, 0.15, 6.0, 0.75),
        # the plain FP64 reference grid (256^2, 10 P_cr, 1 cm steps), a stretch of its 200 steps
        _march("plain-fp64-256", 256, "fp64", 20, 2.56, 0.2, 10.0, 1.0),
        # the sparse grid of the effective-lens method (512^2 over the 8 cm window, 2.5 cm steps), a stretch of its 400
        _march("sparse-512", 512, "fp32", 25, 8.0, 1.0, 100.0, 2.5, diag_every=5),
        # symmetric steps with the exact pointwise substep, the second-order option, on a medium grid
        _march("strang-exact-1024", 1024, "fp32", 13, 8.0, 1.0, 100.0, 0.5, scheme="strang", screen="exact"),
        # an FP64 march of a medium grid, what FP32 runs are checked against
        _march("check-fp64-1024", 1024, "fp64", 5, 8.0, 1.0, 100.0, 0.5),
        # a beam of the statistical ensemble on its own grid, power and peak recorded
        _march("ensemble-2048", 2048, "fp32", 30, 8.0, 1.0, 120.0, 0.5, diag_every=1),
        # the dense-grid problem (4096^2, 8 cm, 1 cm beam at 100 P_cr, 5 mm steps) and its fluence for the sparse fit
        _march("dense-4096", 4096, "fp32", 40, 8.0, 1.0, 100.0, 0.5, diag_every=1, ds=8),
        # the largest grid, a stretch of the 3000-step march of a 3 cm beam at 500 P_cr
        _march("large-8192", 8192, "fp32", 12, 16.0, 3.0, 500.0, 0.5),
        # many uneven beams in one persistent launch, replayed as a graph (mix of 512..2048 as in the 64-beam batch)
        dict(name="ensemble-batch", kind="batch", sizes="2048,512,1024,2048,512,1024,1024,512,2048,512,1024,2048",
             threads=128, steps=10, dz=0.5),
        # the gradient-based fit on the sparse grid through autograd, the first steps of its 400, checkpoint every 20
        dict(name="fit-gradient-512", kind="gradient", api="autograd", n=512, steps=50, ckpt=20, L=8.0, w0=1.0,
             p_cr=100.0, dz=2.5),
        # the large adjoint (8192^2) with few steps per segment
        dict(name="large-gradient-8192", kind="gradient", api="handle", n=8192, steps=6, ckpt=3, L=16.0, w0=3.0,
             p_cr=500.0, dz=0.5),
        # one plane of a filamented cross-section: hot areas, Eq. 8 moments, then a turbulent layer and the lens screen
        dict(name="plane-2048", kind="plane", n=2048, precision="fp32", L=10.24, spots=60, conn=4),
    ]


def draw(rng):
    kind = rng.choice(("march", "march", "march", "march", "batch", "gradient", "plane"))
    if kind == "march":
        precision = rng.choice(("fp32", "fp32", "fp32", "fp64"))
        n = 2 ** rng.randint(6, 13 if precision == "fp32" else 10)
        cap = (12 * 8192 ** 2 if precision == "fp32" else 20 * 1024 ** 2) // (n * n)
        steps = max(1, min(cap, int(round(math.exp(rng.uniform(0.0, math.log(40.5)))))))
        w0 = round(rng.uniform(0.5, 1.5), 3)
        c = _march("", n, precision, steps, round(8.0 * w0, 3), w0, round(rng.uniform(20.0, 150.0), 1),
                   round(rng.uniform(0.3, 0.8), 2), scheme=rng.choice(("lie", "lie", "strang")),
                   screen=rng.choice(("frozen", "frozen", "frozen", "exact")), diag_every=rng.choice((0, 1, 3, 10)),
                   ds=rng.choice((0, 0, 1, 4, 8)))
    elif kind == "batch":
        sizes = [rng.choice((256, 512, 1024, 2048)) for _ in range(rng.randint(2, 14))]
        c = dict(kind="batch", sizes=",".join(str(s) for s in sizes), threads=rng.choice((0, 128, 256)),
                 steps=rng.randint(3, 20), dz=round(rng.uniform(0.3, 0.8), 2))
    elif kind == "gradient":
        n = 2 ** rng.randint(7, 12)
        cap = (6 * 8192 ** 2) // (n * n)
        steps = max(2, min(cap, int(round(math.exp(rng.uniform(math.log(2.0), math.log(60.5)))))))
        c = dict(kind="gradient", api=rng.choice(("autograd", "handle")), n=n, steps=steps,
                 ckpt=rng.randint(1, min(steps, 20)), L=8.0, w0=1.0, p_cr=round(rng.uniform(20.0, 100.0), 1),
                 dz=round(rng.uniform(0.3, 1.0), 2))
    else:
        n = 2 ** rng.randint(8, 11)
        c = dict(kind="plane", n=n, precision=rng.choice(("fp32", "fp32", "fp64")) if n <= 1024 else "fp32",
                 L=round(0.005 * n, 3), spots=rng.randint(5, 60), conn=rng.choice((4, 8)))
    c.pop("name", None)
    return c


# ------------------------------------------------------------------ inputs

def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * int(seed) + salt)
    return g


def _centres(n, L):
    return (torch.arange(n, dtype=torch.float64, device="cuda") - n / 2 + 0.5) * (L / n)


def _noise(n, ell_cells, g):
    """Zero-mean, unit-variance noise, correlated over ell_cells cells."""
    eta = torch.randn((n, n), dtype=torch.float32, device="cuda", generator=g)
    d = torch.arange(n, dtype=torch.float32, device="cuda")
    d = torch.minimum(d, n - d)
    k = torch.fft.fft(torch.exp(-(d * d) / (ell_cells * ell_cells))).real
    eta = torch.fft.irfft2(torch.fft.rfft2(eta) * k[:, None] * k[None, : n // 2 + 1], s=(n, n))
    eta = eta - eta.mean()
    return (eta / eta.std()).double()


def _beam(n, L, w0, p_cr, g, cdtype):
    """Eq. 7 beam of p_cr critical powers, 5 % amplitude noise and 0.1 rad phase
    noise with a correlation of 0.5 mm (at least 3 cells)."""
    x = _centres(n, L)
    ell = max(0.05 / (L / n), 3.0)
    amp = math.sqrt(2.0 * p_cr * configs.critical_power() / (math.pi * w0 * w0))
    gx = torch.exp(-(x * x) / (w0 * w0))
    a = amp * gx[:, None] * gx[None, :] * (1.0 + 0.05 * _noise(n, ell, g))
    ph = 0.1 * _noise(n, ell, g)
    return torch.complex(a * torch.cos(ph), a * torch.sin(ph)).to(cdtype)


def _spots(n, L, spots, g, cdtype):
    """A weak beam carrying hot spots of 2-8 TW/cm^2 with radii of 80-200 um."""
    x = _centres(n, L)
    u = torch.rand((spots, 4), dtype=torch.float64, device="cuda", generator=g)
    w = 5e10 * torch.exp(-(x * x)[:, None] / (0.3 * L) ** 2) * torch.exp(-(x * x)[None, :] / (0.3 * L) ** 2)
    x0, y0 = (u[:, 0] - 0.5) * 0.7 * L, (u[:, 1] - 0.5) * 0.7 * L
    r2 = (0.008 + 0.012 * u[:, 2]) ** 2
    gx = torch.exp(-((x[None, :] - x0[:, None]) ** 2) / r2[:, None])
    gy = torch.exp(-((x[None, :] - y0[:, None]) ** 2) / r2[:, None])
    w = w + (gy * (2e12 + 6e12 * u[:, 3])[:, None]).T @ gx
    ph = 0.3 * torch.sin(2 * math.pi * x / L + 1.0)[None, :] * torch.cos(2 * math.pi * x / L)[:, None]
    a = torch.sqrt(w)
    return torch.complex(a * torch.cos(ph), a * torch.sin(ph)).to(cdtype)


def _cdtype(case):
    return torch.complex128 if case.get("precision") == "fp64" else torch.complex64


def _physics(case, n=None, L=None):
    """Workload dict of a case: the full screen, or Kerr alone for the plane."""
    terms = configs.KERR | configs.DIFFRACTION if case["kind"] == "plane" else configs.ALL_TERMS
    cfg = configs.physics(n or case["n"], L or case["L"], case.get("dz", 0.5), terms,
                          theta=GAINS if case["kind"] == "gradient" else configs.NOMINAL_THETA)
    cfg.update(scheme=case.get("scheme", "lie"), screen=case.get("screen", "frozen"))
    return cfg


def _batch_beams(case, seed):
    """(n, L, w0, P / P_cr) and the input field of every beam."""
    g = torch.Generator()
    g.manual_seed(int(seed) + 77)
    for b, n in enumerate(int(s) for s in case["sizes"].split(",")):
        u = torch.rand(2, dtype=torch.float64, generator=g)
        w0, p = 0.5 + float(u[0]), 20.0 + 180.0 * float(u[1])
        yield n, 8.0 * w0, _beam(n, 8.0 * w0, w0, p, _gen(seed, b), torch.complex64)


def _target(case, seed):
    """Target fluence of a fit: the input plane of another beam, slightly wider."""
    v = _beam(case["n"], case["L"], 1.05 * case["w0"], case["p_cr"], _gen(seed, 5), torch.complex64)
    return (v.real.double() ** 2 + v.imag.double() ** 2).contiguous()


def _draws(case, seed):
    n, cdt = case["n"], _cdtype(case)
    return torch.randn((n, n), dtype=cdt, device="cuda", generator=_gen(seed, 3))


# turbulent layer: one metre of eps_t with structure down to 2 mm, about 0.5 rad of phase
K_H, THICKNESS, TURB_RAD = 30.0, 100.0, 0.5


def _tau(case):
    k0 = 2.0 * math.pi * configs.N0 / configs.LAMBDA0
    bins = max(1.0, math.pi * (K_H * case["L"] / (2.0 * math.pi)) ** 2)
    return TURB_RAD * 2.0 * k0 / THICKNESS / math.sqrt(0.5 * bins)


W_HOT, PQ = 1.0e12, [(1, 1), (1, 0), (2, 2)]


# ------------------------------------------------------------------- cases

def prepare(case, seed):
    kind = case["kind"]
    if kind == "march":
        U = _beam(case["n"], case["L"], case["w0"], case["p_cr"], _gen(seed, 0), _cdtype(case))
        return dict(case=case, U=U, g=Grid(_physics(case), precision=case["precision"], diag_every=case["diag_every"]))
    if kind == "batch":
        fields = list(_batch_beams(case, seed))
        b = Batch([_physics(case, n, L) for n, L, _ in fields], {"threads": case["threads"]} if case["threads"] else None)
        for i, (_, _, U) in enumerate(fields):
            b.load(i, U)
        return dict(case=case, b=b.capture(case["steps"]), count=len(fields))
    if kind == "gradient":
        U = _beam(case["n"], case["L"], case["w0"], case["p_cr"], _gen(seed, 0), torch.complex64)
        fit = AdjointMarch(_physics(case), case["steps"], case["ckpt"], precision="fp32")
        D = _target(case, seed)
        st = dict(case=case, U=U, fit=fit, D=D)
        if case["api"] == "autograd":
            st.update(theta=torch.tensor(GAINS, dtype=torch.float32, requires_grad=True), U=U.requires_grad_(True))
        else:
            fit.set_target(D)
        return st
    g = Grid(_physics(case), precision=case["precision"])
    return dict(case=case, g=g, U=_spots(case["n"], case["L"], case["spots"], _gen(seed, 0), _cdtype(case)),
                xi=_draws(case, seed))


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "march":
        g = st["g"]
        g.load(st["U"]).step(case["steps"])
        out = {"field": g.field(device=True)}
        if case["ds"]:
            out["fluence"] = g.fluence(case["ds"], device=True)
        if case["diag_every"]:
            power, peak = g.history()
            out["power"], out["peak"] = power.astype(g.rdtype), peak.astype(g.rdtype)
        return out
    if kind == "batch":
        b = st["b"].replay()
        return [b.field(i, device=True) for i in range(st["count"])]
    if kind == "gradient":
        if case["api"] == "autograd":
            st["theta"].grad = st["U"].grad = None
            loss = NlseFluenceLoss.apply(st["theta"], st["U"], st["D"], st["fit"])
            loss.backward()
            return {"loss": float(loss), "theta": st["theta"].grad, "U0": st["U"].grad}
        loss = st["fit"].forward(st["U"])
        dth, dU = st["fit"].backward()
        return {"loss": loss, "theta": dth.astype(np.float32), "U0": dU}
    g = st["g"]
    g.load(st["U"])
    count, labels = g.hot_areas(W_HOT, case["conn"], labels=True, device=True)
    moments = g.moments(PQ).astype(g.rdtype)
    g.turbulent_screen(st["xi"], _tau(case), K_H, THICKNESS)
    lenses, centres, w_dif = g.effective_lens(dict(LENS, conn=case["conn"]), w_dif=True)
    listed_centres = np.full(case["spots"], -1, dtype=np.int32)  # at most one lens per spot
    listed_centres[:lenses] = centres
    return {"count": count, "labels": labels, "moments": moments, "lenses": lenses, "centres": listed_centres,
            "w_dif": w_dif, "field": g.field(device=True)}


def work(case):
    """Bytes: inputs and outputs once, and for every step two sweeps of the
    field (a 2D transform of a grid larger than one SM needs every row and then
    every column, so each of a step's two passes reads and writes the field).
    Flops: 5 N log2 N per transform of N points, about 50 per point for the
    propagator and the screen."""
    kind = case["kind"]
    cs = 16 if case.get("precision") == "fp64" else 8

    def step(n):
        return 10.0 * n * n * math.log2(n * n) + 50.0 * n * n

    if kind == "march":
        nn = case["n"] ** 2
        out = cs * nn + (cs // 2 * nn / case["ds"] ** 2 if case["ds"] else 0)
        sweeps = case["steps"] + (0.5 if case["scheme"] == "strang" else 0)  # the opening half screen
        return {"bytes": cs * nn + out + 4.0 * cs * nn * sweeps, "flops": step(case["n"]) * case["steps"]}
    if kind == "batch":
        ns = [int(s) for s in case["sizes"].split(",")]
        return {"bytes": sum(n * n * (8.0 + 32.0 * case["steps"]) for n in ns),
                "flops": sum(step(n) for n in ns) * case["steps"]}
    if kind == "gradient":
        # the forward march (with a stored checkpoint per segment), the march of every segment again with its
        # fields stored, and the backward sweep, whose row pass reads a stored field beside the adjoint's
        n, s = case["n"], case["steps"]
        return {"bytes": n * n * (8.0 + 8.0 + 16.0 + 32.0 * s + 40.0 * s + 40.0 * s + 16.0 * math.ceil(s / case["ckpt"])),
                "flops": 3.25 * step(n) * s}
    nn = case["n"] ** 2
    # the field and the draws in, the labels, w_dif and the field out
    return {"bytes": nn * (cs + cs + 4.0 + cs / 2 + cs), "flops": 8.0 * step(case["n"])}


# ------------------------------------------- the same in plain 64-bit torch

def _coef(cfg, dz):
    k0 = 2.0 * math.pi * cfg["n0"] / cfg["lambda0"]
    eps_k = 2.0 * k0 * k0 * cfg["n2"] / cfg["n0"]
    eps_m = -k0 * k0 * cfg["sigmaK"] * cfg["rho_nt"] * cfg["tau_pl"] / cfg["rho_c"]
    on = [1.0 if cfg["terms"] & t else 0.0 for t in (configs.KERR, configs.PLASMA, configs.MPA)]
    # exponents per W/cm^2 (Kerr), (W/cm^2)^K scaled to 1e13 W/cm^2 (plasma), and absorption
    return (on[0] * dz * eps_k / (2.0 * k0), on[1] * dz * eps_m / (2.0 * k0) * 1e13 ** cfg["K"],
            -on[2] * dz * cfg["betaK"] / 2.0 * 1e13 ** (cfg["K"] - 1))


def _exact_screen(v, cfg, dz, theta):
    """v exp(s(|v|^2)), or the closed-form pointwise substep."""
    aK, aP, aA = _coef(cfg, dz)
    K = cfg["K"]
    I = v.real ** 2 + v.imag ** 2
    u = I / 1e13
    u2 = u * u
    u4 = u2 * u2
    u7 = u4 * u2 * u
    assert K == 8
    if cfg["screen"] == "exact":
        a = -2.0 * (K - 1) * theta[4] * aA * u7
        ok = a > 0
        l = torch.log1p(a)
        e = (K - 2) / (K - 1)
        safe = torch.where(ok, a, torch.ones_like(a))
        f1 = torch.where(ok, torch.expm1(e * l) / (safe * e), torch.ones_like(a))
        fk = torch.where(ok, -(K - 1) * torch.expm1(-l / (K - 1)) / safe, torch.ones_like(a))
        ph = -theta[0] * aK * I * f1 - theta[2] * aP * u4 * u4 * fk
        amp = torch.exp(-l / (2 * (K - 1)))
        return v * torch.complex(amp * torch.cos(ph), amp * torch.sin(ph))
    re = theta[1] * aK * I + theta[3] * aP * (u4 * u4) + theta[4] * aA * u7
    im = -theta[0] * aK * I - theta[2] * aP * (u4 * u4) + theta[5] * aA * u7
    return v * torch.exp(torch.complex(re, im))


def _propagator(cfg):
    n = cfg["n"]
    k0 = 2.0 * math.pi * cfg["n0"] / cfg["lambda0"]
    k = 2.0 * math.pi * torch.fft.fftfreq(n, cfg["L"] / n, dtype=torch.float64, device="cuda")
    ph = k * k * cfg["dz"] / (2.0 * k0)
    return torch.polar(torch.ones_like(ph), ph)


def _exact_march(U, cfg, steps, theta, diag_every=0):
    p = _propagator(cfg)
    strang = cfg["scheme"] == "strang"
    h = cfg["dz"] * (0.5 if strang else 1.0)
    rec = []
    for s in range(steps):
        if strang:
            U = _exact_screen(U, cfg, h, theta)
        U = torch.fft.ifft2(torch.fft.fft2(U) * p[:, None] * p[None, :])
        U = _exact_screen(U, cfg, h, theta)
        if diag_every and (s + 1) % diag_every == 0:
            I = U.real ** 2 + U.imag ** 2
            rec.append((float(I.sum()) * (cfg["L"] / cfg["n"]) ** 2, float(I.max())))
    return U, rec


def _exact_gradient(case, seed):
    cfg = _physics(case)
    U = _beam(case["n"], case["L"], case["w0"], case["p_cr"], _gen(seed, 0), torch.complex64).to(torch.complex128)
    D = _target(case, seed)
    # gains as the case passes them: FP32 leaves through autograd, FP64 in the handle's parameters
    dt = torch.float32 if case["api"] == "autograd" else torch.float64
    theta = torch.tensor(GAINS, dtype=dt).double()
    # the recorded graph of one segment at a time: fields at the segment starts, then backwards
    seg = max(1, min(case["steps"], int(4e9 / (16.0 * case["n"] ** 2)), 16))
    starts = []
    with torch.no_grad():
        V = U
        for s in range(0, case["steps"], seg):
            starts.append(V)
            V, _ = _exact_march(V, cfg, min(seg, case["steps"] - s), theta.tolist())
        F = V.real ** 2 + V.imag ** 2
        S = float((D * D).sum())
        loss = float(((F - D) ** 2).sum()) / S
        G = 4.0 * (F - D) / S * V
    dth = torch.zeros(6, dtype=torch.float64)
    for i in reversed(range(len(starts))):
        m = min(seg, case["steps"] - i * seg)
        U0 = starts[i].detach().requires_grad_(True)
        th = theta.cuda().clone().requires_grad_(True)
        V, _ = _exact_march(U0, cfg, m, th)
        (torch.conj(G) * V).real.sum().backward()
        G = U0.grad
        dth += th.grad.cpu()
    return {"loss": loss, "theta": dth, "U0": G}


def _regions(mask, conn):
    """Smallest row-major index of every pixel's connected region (n n outside)."""
    n = mask.shape[0]
    far = n * n
    lab = torch.where(mask, torch.arange(far, device=mask.device).view(n, n), far)
    for _ in range(4 * n):
        pad = torch.nn.functional.pad(lab, (1, 1, 1, 1), value=far)
        near = [pad[1 + dy:n + 1 + dy, 1 + dx:n + 1 + dx] for dy in (-1, 0, 1) for dx in (-1, 0, 1)
                if (dy or dx) and (conn == 8 or not (dy and dx))]
        new = lab
        for x in near:
            new = torch.minimum(new, x)
        new = torch.where(mask, new, far)
        if torch.equal(new, lab):
            break
        lab = new
    return lab


def _exact_plane(case, seed):
    n, L = case["n"], case["L"]
    U = _spots(n, L, case["spots"], _gen(seed, 0), _cdtype(case)).to(torch.complex128)
    I = U.real ** 2 + U.imag ** 2
    x = _centres(n, L)
    r2 = (x * x)[:, None] + (x * x)[None, :]
    moments = [float((I ** p * r2 ** q).sum()) * (L / n) ** 2 for p, q in PQ]
    m = torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device="cuda").round()
    disc = (m * m)[:, None] + (m * m)[None, :] <= (K_H * L / (2.0 * math.pi)) ** 2
    eps = torch.fft.ifft2(_draws(case, seed).to(torch.complex128) * disc).real * (_tau(case) * n * n)
    k0 = 2.0 * math.pi * configs.N0 / configs.LAMBDA0
    U = U * torch.exp(-1j * THICKNESS * eps / (2.0 * k0))
    k2 = (2.0 * math.pi / L * m) ** 2
    w = U.real ** 2 + U.imag ** 2
    w = torch.fft.ifft2(torch.fft.fft2(w) * torch.exp(-LENS["l_dif"] * (k2[:, None] + k2[None, :]))).real
    lab = _regions(w >= LENS["w_l"], case["conn"])
    idx = torch.nonzero((lab < n * n).view(-1)).view(-1)
    dre, dim = torch.zeros_like(w), torch.zeros_like(w)
    labs, vals = lab.view(-1)[idx], w.view(-1)[idx]
    for root in torch.unique(labs).tolist():
        sel = labs == root
        c = int(idx[sel][torch.argmax(vals[sel])])
        r = torch.sqrt((x - x[c // n])[:, None] ** 2 + (x - x[c % n])[None, :] ** 2)
        for acc, part in ((dre, LENS["re"]), (dim, LENS["im"])):
            inner = 0.0
            for (rj, a, om, ps) in part:
                acc += torch.where((r >= inner) & (r < rj), a * torch.cos(om * r + ps), torch.zeros_like(r))
                inner = rj
    return {"count": None, "labels": None, "moments": np.array(moments), "lenses": None, "centres": None, "w_dif": w,
            "field": U * torch.exp(torch.complex(-dim, dre))}


def exact(case, seed):
    kind = case["kind"]
    if kind == "march":
        cfg = _physics(case)
        U = _beam(case["n"], case["L"], case["w0"], case["p_cr"], _gen(seed, 0), _cdtype(case)).to(torch.complex128)
        U, rec = _exact_march(U, cfg, case["steps"], cfg["theta"], case["diag_every"])
        out = {"field": U}
        if case["ds"]:
            m = case["n"] // case["ds"]
            F = U.real ** 2 + U.imag ** 2
            out["fluence"] = F.view(m, case["ds"], m, case["ds"]).mean(dim=(1, 3))
        if case["diag_every"]:
            out["power"] = np.array([r[0] for r in rec])
            out["peak"] = np.array([r[1] for r in rec])
        return out
    if kind == "batch":
        out = []
        for n, L, U in _batch_beams(case, seed):
            cfg = _physics(case, n, L)
            out.append(_exact_march(U.to(torch.complex128), cfg, case["steps"], cfg["theta"])[0])
        return out
    if kind == "gradient":
        return _exact_gradient(case, seed)
    return _exact_plane(case, seed)
