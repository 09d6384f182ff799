"""Performance cases of the focal-field evaluator.

Each case is one call that a user's program makes through the package's
public entry points (``Context.eval``, ``eval_time_domain``, ``time_domain``,
``eval_batch``) with the context, mirror, beam and observation points it holds
already.  Lengths are in lambda0, omegas in units of omega0; mirrors have
r_max = 2 f and beams w0 = 0.6 f, as in the package's workloads.

``exact`` restates the sums in 64 bits with plain torch: the quadrature of the
physical-optics Stratton-Chu integrals (Eq. 11 of arXiv:1609.08146) over the
paraboloid, its rim line integral, and the inverse transform of Eq. 13.
"""
import math

import numpy as np
import torch

import paper_1609_08146_gb300 as sc

_BASE = dict(kind="eval", f=62500.0, r_min=0.0, n_r=128, n_theta=128, radial="gauss_legendre", profile="gauss",
             pol="linear", n_zernike=0, n_omega=1, n_points=1024, layout="cube", precision="fp32", host=False)


def _case(name, **kw):
    return dict(_BASE, name=name, **kw)


def listed():
    return [
        # one frequency on a small focal plane: the smallest call of an interactive session or a parameter scan
        _case("mono_small", f=20.0, n_r=64, n_theta=64, layout="plane"),
        # the same plane in the plain FP64 form, the check a user runs beside the fast path
        _case("mono_small_fp64", f=20.0, n_r=64, n_theta=64, layout="plane", precision="fp64"),
        # a fine monochromatic intensity map of a radially polarised focus
        _case("mono_map", f=1e4, n_r=256, n_theta=256, n_points=65536, layout="plane", pol="radial"),
        # a handful of laser lines on an annular, aberrated mirror, ragged sizes, numpy in and numpy out
        _case("few_lines_host", f=5e3, r_min=750.0, n_r=129, n_theta=200, radial="simpson", pol="azimuthal",
              profile="supergauss", n_zernike=14, n_omega=11, n_points=3001, host=True),
        # a many-cycle pulse: a few dozen frequencies on a focal cube
        _case("narrow_band", f=1e3, n_r=256, n_theta=256, n_omega=48, n_points=4096),
        # the headline workload: a 10 fs pulse, 256 frequencies, 512 x 512 nodes, a focal plane and the axis
        _case("broadband", n_r=512, n_theta=512, n_omega=256, n_points=4160, layout="plane"),
        # a ragged broadband request: odd counts everywhere, aberrated super-Gaussian radial beam
        _case("ragged_band", f=3e3, n_r=200, n_theta=190, n_omega=100, n_points=1531, pol="radial",
              profile="supergauss", n_zernike=14),
        # a finely sampled spectrum on a coarse mirror: the largest frequency counts
        _case("fine_band", f=1e5, n_r=128, n_theta=128, n_omega=512, n_points=1024),
        # a broadband check in the plain FP64 form
        _case("band_fp64", f=1e4, n_omega=64, n_points=512, precision="fp64"),
        # inverse transform of stored spectra to 512 time samples (movies of the focal field)
        _case("transform", kind="transform", n_omega=256, n_points=4160, n_t=512),
        # a vortex pulse straight to the time domain (Laguerre-Gauss beam, several node tables)
        _case("pulse_vortex", kind="pulse", f=1e3, n_r=96, n_theta=96, profile="laguerre_gauss", n_omega=96,
              n_points=600, n_t=201),
        # a mixed queue of uneven requests evaluated together
        _case("batch", kind="batch", n_requests=24, max_side=256, max_points=8192, max_omega=256),
    ]


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _logi(rng, lo, hi):
    return int(round(_logu(rng, lo, hi)))


def draw(rng):
    kind = rng.choice(["eval"] * 5 + ["fp64", "transform", "pulse", "batch"])
    c = dict(_BASE)
    if kind == "transform":
        while True:
            c.update(kind="transform", n_omega=_logi(rng, 8, 512), n_points=_logi(rng, 64, 16384),
                     n_t=_logi(rng, 33, 1024))
            if c["n_omega"] * c["n_points"] * c["n_t"] <= 2e9:
                return c
    if kind == "batch":
        c.update(kind="batch", n_requests=_logi(rng, 4, 24), max_side=rng.choice([64, 128, 256]),
                 max_points=_logi(rng, 512, 8192), max_omega=_logi(rng, 8, 256))
        return c
    fp64 = kind == "fp64"
    limit = 5e8 if fp64 else 1e10 if kind == "pulse" else 3e10
    while True:
        c.update(f=_logu(rng, 20.0, 1e5), n_r=_logi(rng, 33, 512), n_theta=_logi(rng, 32, 512),
                 n_omega=_logi(rng, 1, 512), n_points=_logi(rng, 64, 65536), layout=rng.choice(["cube", "plane"]),
                 profile=rng.choice(["gauss", "gauss", "supergauss", "tophat"]),
                 pol=rng.choice(["linear", "radial", "azimuthal"]), n_zernike=rng.choice([0, 0, 4, 14]))
        c["r_min"] = rng.choice([0.0, 0.0, 0.15]) * c["f"]
        c["radial"] = rng.choice(["gauss_legendre", "gauss_legendre", "simpson"])
        if c["radial"] == "simpson":
            c["n_r"] |= 1
        if 1e6 <= _evals(c) <= limit:
            break
    if fp64:
        c["precision"] = "fp64"
    elif kind == "pulse":
        c.update(kind="pulse", n_omega=max(4, min(c["n_omega"], 256)), n_points=min(c["n_points"], 4096),
                 n_t=_logi(rng, 33, 512))
        if rng.random() < 0.5 and c["f"] >= 300.0:
            c.update(profile="laguerre_gauss", pol="linear")
    else:
        c["host"] = rng.random() < 0.2
    return c


def _evals(c):
    return float(c["n_r"]) * c["n_theta"] * c["n_omega"] * c["n_points"]


# ---------------------------------------------------------------- inputs


def _omegas(n):
    return np.array([1.0]) if n == 1 else np.linspace(0.5, 1.5, n)


def _points(c, rng):
    n = c["n_points"]
    if c["layout"] == "cube":
        return rng.uniform(-2.0, 2.0, size=(n, 3))
    # the largest square grid over +-3 in a slightly displaced plane, the rest along the axis
    s = math.isqrt(n)
    g = np.linspace(-3.0, 3.0, s)
    x, y = np.meshgrid(g, g, indexing="ij")
    p = np.zeros((n, 3))
    p[:s * s, 0], p[:s * s, 1] = x.ravel(), y.ravel()
    p[s * s:, 2] = np.linspace(-5.0, 5.0, n - s * s)
    return p + rng.uniform(-0.05, 0.05, size=3)


def _beam(c, rng):
    """Beam, spectrum amplitudes and aberrations of one request."""
    om = _omegas(c["n_omega"])
    amp = np.exp(-((om - 1.0) / 0.3) ** 2) * np.exp(1j * rng.normal(0.0, 10.0) * (om - 1.0) ** 2)
    b = dict(profile=c["profile"], w0=0.6 * c["f"], sg_order=4, pol=c["pol"],
             zernike=[float(v) for v in rng.normal(0.0, 0.1, size=c["n_zernike"])])
    if c["pol"] == "linear":
        b["pol_angle"] = float(rng.uniform(0.0, math.pi))
    if c["profile"] == "laguerre_gauss":
        b.update(lg_p=0, lg_l=1, z_waist=-0.5 * c["f"])
    return om, amp, b


def _request(c, rng):
    om, amp, b = _beam(c, rng)
    return dict(c, omegas=om, amp=amp, beam=b, points=_points(c, rng))


def _requests(c, seed):
    """The requests of a case: inputs made from the seed alone."""
    rng = np.random.Generator(np.random.PCG64([seed, 1609]))
    if c["kind"] != "batch":
        return [_request(c, rng)]
    # shapes from the case, as uneven as a serving mix; values from the seed
    shp = np.random.Generator(np.random.PCG64([c["n_requests"], c["max_side"], c["max_points"], c["max_omega"]]))
    out = []
    for _ in range(c["n_requests"]):
        side = int(shp.choice([s for s in (64, 128, 256) if s <= c["max_side"]]))
        r = dict(_BASE, f=float(10 ** shp.uniform(3, 5)), n_r=side, n_theta=side,
                 profile=str(shp.choice(["gauss", "supergauss"])),
                 pol=str(shp.choice(["linear", "radial", "azimuthal"])), n_zernike=14,
                 n_points=int(round(10 ** shp.uniform(math.log10(256), math.log10(c["max_points"])))),
                 n_omega=int(round(10 ** shp.uniform(0, math.log10(c["max_omega"])))))
        out.append(_request(r, rng))
    return out


def _times(c):
    return (np.arange(c["n_t"]) - c["n_t"] // 2) / 8.0


def _spectra(c, seed):
    """Stored spectra E, B [n_omega, n_points, 3]: a pulse's envelope in omega, speckle in space."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    om = _omegas(c["n_omega"])
    env = torch.tensor(np.exp(-((om - 1.0) / 0.3) ** 2), dtype=torch.float32, device="cuda")[:, None, None, None]
    out = []
    for _ in range(2):
        r = torch.randn((c["n_omega"], c["n_points"], 3, 2), generator=gen, device="cuda")
        out.append(torch.view_as_complex(r * env))
    return out


def prepare(case, seed):
    ctx = sc.Context(0)
    if case["kind"] == "transform":
        E, B = _spectra(case, seed)
        return dict(case=case, ctx=ctx, E=E, B=B, omegas=_omegas(case["n_omega"]), times=_times(case))
    reqs = []
    for r in _requests(case, seed):
        m = ctx.mirror(r["f"], r["r_min"], 2 * r["f"], r["n_r"], r["n_theta"], rim=True, radial=r["radial"])
        kw = dict(r["beam"], omega_band=(0.5, 1.5)) if r["profile"] == "laguerre_gauss" else r["beam"]
        inc = ctx.incident(spectrum=dict(kind="sampled", omega=r["omegas"], amp=r["amp"]), **kw)
        pts = r["points"] if r["host"] else torch.tensor(r["points"], dtype=torch.float64, device="cuda")
        reqs.append((m, inc, r["omegas"], pts))
    return dict(case=case, ctx=ctx, reqs=reqs, times=_times(case) if case["kind"] == "pulse" else None)


def run(state):
    c, ctx = state["case"], state["ctx"]
    if c["kind"] == "transform":
        return ctx.time_domain(state["E"], state["B"], state["omegas"], state["times"])
    if c["kind"] == "batch":
        return ctx.eval_batch(state["reqs"])
    m, inc, om, pts = state["reqs"][0]
    if c["kind"] == "pulse":
        return ctx.eval_time_domain(m, inc, om, pts, state["times"])
    return ctx.eval(m, inc, om, pts, precision=c["precision"])


def work(case):
    """One (point, node, omega) term: one complex phase factor from the last (8 flops) and nine complex-by-real
    multiply-adds (36); one (point, node) pair: its geometry and coefficients (about 60).  A transform term: one
    complex multiply-add's real part (4)."""
    c = case
    if c["kind"] == "transform":
        n = 2.0 * 3 * c["n_points"]
        return dict(bytes=n * (8.0 * c["n_omega"] + 4.0 * c["n_t"]), flops=4.0 * n * c["n_omega"] * c["n_t"])
    by = fl = 0.0
    for r in _requests(c, 0):
        elem = 16 if r["precision"] == "fp64" else 8
        nodes, np_, no = float(r["n_r"] * r["n_theta"]), r["n_points"], r["n_omega"]
        by += 24.0 * np_ + (9 * elem / 2) * nodes
        fl += np_ * nodes * (60.0 + 44.0 * no)
        by += 2.0 * 3 * np_ * (4 * c["n_t"] if c["kind"] == "pulse" else elem * no)
        if c["kind"] == "pulse":
            fl += 4.0 * 6 * np_ * no * c["n_t"]
    return dict(bytes=by, flops=fl)


# ---------------------------------------------------------------- 64-bit restatement


def _noll(j):
    n = int((math.sqrt(8 * j - 7) - 1) / 2)
    k = j - n * (n + 1) // 2 - 1  # 0-based position in row n
    m = 2 * ((k + 1) // 2) if n % 2 == 0 else 2 * (k // 2) + 1
    return n, m if j % 2 == 0 else -m


def _zernike(j, u, th):
    n, m = _noll(j)
    a = abs(m)
    R = np.zeros_like(u)
    for s in range((n - a) // 2 + 1):
        R += ((-1) ** s * math.factorial(n - s) / (math.factorial(s) * math.factorial((n + a) // 2 - s)
                                                   * math.factorial((n - a) // 2 - s))) * u ** (n - 2 * s)
    if m == 0:
        return math.sqrt(n + 1) * R
    return math.sqrt(2 * (n + 1)) * R * (np.cos(a * th) if m > 0 else np.sin(a * th))


def _radial(c):
    a, b, n = c["r_min"], 2 * c["f"], c["n_r"]
    if c["radial"] == "simpson":
        w = np.full(n, 2.0)
        w[1::2], w[0], w[-1] = 4.0, 1.0, 1.0
        return np.linspace(a, b, n), w * (b - a) / (n - 1) / 3.0
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (b + a) + 0.5 * (b - a) * x, 0.5 * (b - a) * w


def _e_perp(r, rho, th, z, k):
    """Transverse incident field (complex) at mirror points, without its plane phase and aberration."""
    b, w0 = r["beam"], r["beam"]["w0"]
    if b["profile"] == "laguerre_gauss":
        zr, zeta, a = 0.5 * k * w0 * w0, b["z_waist"] - z, abs(b["lg_l"])
        w2 = w0 * w0 * (1.0 + (zeta / zr) ** 2)
        u = (w0 * w0 / w2) ** (0.5 * (a + 1)) * (rho / w0) ** a * np.exp(-rho * rho / w2)
        u = u * np.exp(1j * (0.5 * k * rho * rho * zeta / (zeta * zeta + zr * zr) - (a + 1) * np.arctan(zeta / zr)
                             + b["lg_l"] * th))
        return u * math.cos(b["pol_angle"]), u * math.sin(b["pol_angle"])
    if b["profile"] == "gauss":
        A = np.exp(-(rho / w0) ** 2)
    elif b["profile"] == "supergauss":
        A = np.exp(-(rho / w0) ** (2 * b["sg_order"]))
    else:
        A = np.where(rho <= w0, 1.0, 0.0)
    if b["pol"] == "linear":
        return A * math.cos(b["pol_angle"]), A * math.sin(b["pol_angle"])
    A = A * rho / w0
    return (A * np.cos(th), A * np.sin(th)) if b["pol"] == "radial" else (-A * np.sin(th), A * np.cos(th))


def _nodes(r):
    """Surface and rim points (rho, theta, weight, side of the rim or 0)."""
    th = 2 * math.pi * np.arange(r["n_theta"]) / r["n_theta"]
    x, w = _radial(r)
    dth = 2 * math.pi / r["n_theta"]
    rho, t = np.repeat(x, th.size), np.tile(th, x.size)
    wq, side = np.repeat(w * x, th.size) * dth, np.zeros(rho.size)
    for edge, s in ((2 * r["f"], 1.0), (r["r_min"], -1.0)):
        if edge > 0.0:
            rho, t = np.append(rho, np.full(th.size, edge)), np.append(t, th)
            wq, side = np.append(wq, np.full(th.size, edge * dth)), np.append(side, np.full(th.size, s))
    return rho, t, wq, side


def _sources(r, rho, t, z, wq, side, k):
    """J and rho per node: N x B~ and N . E~ times the weight over 2 pi; on the rim the conormal current alone."""
    ex, ey = _e_perp(r, rho, t, z, k)
    Nx, Ny = -rho * np.cos(t) / (2 * r["f"]), -rho * np.sin(t) / (2 * r["f"])
    bx, by = ey, -ex
    J = np.stack([-by, bx + 0 * Nx, Nx * by - Ny * bx])
    q = side * (J[0] * np.cos(t) + J[1] * np.sin(t) + J[2] * rho / (2 * r["f"])) / (1.0 + (rho / (2 * r["f"])) ** 2)
    surf = side == 0
    return np.where(surf, J, 0.0) * wq / (2 * math.pi), np.where(surf, Nx * ex + Ny * ey, q) * wq / (2 * math.pi)


def _field(r):
    """E, B [n_omega, n_points, 3] complex128."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    rho, t, wq, side = _nodes(r)
    f = r["f"]
    z = rho * rho / (4 * f) - f
    W = sum((a * _zernike(i + 2, rho / (2 * f), t) for i, a in enumerate(r["beam"]["zernike"])), np.zeros_like(rho))
    to = lambda a: torch.tensor(np.ascontiguousarray(a), device=dev)
    P = to(np.stack([rho * np.cos(t), rho * np.sin(t), z], axis=1))
    pn, Wt, rim = to(z + 2 * f), to(W), to(side != 0)
    pts = to(r["points"])
    n_om, n_p = len(r["omegas"]), pts.shape[0]
    E = torch.empty((n_om, n_p, 3), dtype=torch.complex128, device=dev)
    B = torch.empty_like(E)
    fixed = r["beam"]["profile"] != "laguerre_gauss"
    step = max(1, int(4e7) // P.shape[0])
    src = []
    for om in r["omegas"]:
        if not (fixed and src):
            J, q = _sources(r, rho, t, z, wq, side, 2 * math.pi * om)
            J, q = to(J.T.astype(np.complex128)), to(q.astype(np.complex128))
            Pc = P.to(torch.complex128)
            JP = torch.linalg.cross(J, Pc)
            src.append((J, torch.cat([JP, J], 1), torch.cat([q[:, None] * Pc, q[:, None]], 1)))
    for p0 in range(0, n_p, step):
        x = pts[p0:p0 + step]
        d2 = (P[None, :, 0] - x[:, None, 0]) ** 2
        d2 += (P[None, :, 1] - x[:, None, 1]) ** 2
        d2 += (P[None, :, 2] - x[:, None, 2]) ** 2
        R = d2.sqrt_()
        # R - |P| without the cancellation
        phi = ((x * x).sum(1)[:, None] - 2.0 * (x @ P.T)) / (R + pn) + Wt
        iR = 1.0 / R
        xc = x.to(torch.complex128)
        for i, om in enumerate(r["omegas"]):
            k = 2 * math.pi * om
            J, JB, Q = src[0 if fixed else i]
            G = torch.polar(iR, k * phi)
            e = 1j * k * (G @ J)
            A = torch.complex(-iR, torch.full_like(iR, k)) * G * iR
            s = A @ JB
            b = s[:, :3] - torch.linalg.cross(s[:, 3:], xc)
            A = torch.where(rim, A * (1j / k), A)
            s = A @ Q
            e = e + s[:, :3] - s[:, 3:] * xc
            a = complex(r["amp"][i])
            E[i, p0:p0 + step], B[i, p0:p0 + step] = a * e, a * b
    return E, B


def _transform(F, omegas, times):
    k = torch.tensor(2 * math.pi * omegas, device=F.device)
    dk = 2 * math.pi * (omegas[-1] - omegas[0]) / (len(omegas) - 1) if len(omegas) > 1 else 1.0
    ph = torch.outer(torch.tensor(times, device=F.device), k)
    M = torch.polar(torch.ones_like(ph), -ph)
    n_p = F.shape[1]
    F = F.to(torch.complex128).reshape(F.shape[0], -1)
    return (2.0 * dk * (M.real @ F.real - M.imag @ F.imag)).reshape(len(times), n_p, 3)


def exact(case, seed):
    if case["kind"] == "transform":
        E, B = _spectra(case, seed)
        return tuple(_transform(F, _omegas(case["n_omega"]), _times(case)) for F in (E, B))
    reqs = _requests(case, seed)
    if sum(_evals(r) for r in reqs) > 2e10:
        return None
    if case["kind"] == "pulse":
        return tuple(_transform(F, reqs[0]["omegas"], _times(case)) for F in _field(reqs[0]))
    out = [_field(r) for r in reqs]
    if case["kind"] == "batch":
        return out
    return tuple(F.cpu().numpy() for F in out[0]) if case["host"] else out[0]
