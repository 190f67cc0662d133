"""The work that programs have this library do, as cases that can be timed.

A program of the discrete dipole approximation sets a target and its materials,
prepares a wavelength, solves A P = E for its incident waves, and derives
efficiencies, scattered fields and gradients from P.  ``listed`` names twelve
such calls, from one small product A x to a sweep of sixty-four right-hand
sides and a product on the largest lattice; ``draw`` gives more of the same
kinds over the range of lattices, right-hand sides, precisions and options
that users bring.  ``prepare`` makes what a program has in hand before the
call, ``run`` is the call, ``work`` what it cannot do without, and ``exact``
its result by plain FFTs and BiCGstab in 64 bits.

Results of the complex64 modes are kept in complex64 (float32 for the
efficiencies): that is the accuracy their arithmetic or the solve's tolerance
gives them, whatever type the call widens them to.
"""
import math

import numpy as np
import torch

import paper_1202_3424_gb300 as dda
from paper_1202_3424_gb300.autograd import DipoleTarget, QabsFn

PREC = {"fp64": dda.Precision.FP64, "refined": dda.Precision.FP32_REFINED, "fp32": dda.Precision.FP32,
        "df64": dda.Precision.DF64}


def _case(kind, name=None, **kw):
    c = {"kind": kind, "shape": "ellipsoid", "nx": 32, "ny": 32, "nz": 32, "m_re": 1.33, "m_im": 0.01, "x": 1.0, "R": 2,
         "prec": "refined", "tol": 1e-5, "solver": "bicgstab", "materials": "one", "products": 60}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one product on the small lattice, as a program with its own iteration calls it: launches and host path
        _case("matvec", "product_small", nx=16, ny=16, nz=16, x=1.0, R=1, prec="fp32"),
        # odd, unequal sides and a few right-hand sides: the padded lengths are 128, 96 and 64 points
        _case("matvec", "product_ragged", nx=53, ny=41, nz=29, x=3.0, R=6, prec="fp32"),
        # the largest lattice the library takes
        _case("matvec", "product_large", nx=256, ny=256, nz=256, x=20.0, R=4, prec="fp32"),
        # the accurate residual of a program that refines by itself
        _case("matvec", "product_accurate", nx=96, ny=64, nz=32, m_im=0.05, x=8.0, R=8, prec="df64"),
        # one wavelength of a spectrum: materials, Green tensor and both polarizations of a small grain
        _case("spectrum", "spectrum_step", nx=24, ny=24, nz=24, m_re=1.6, m_im=0.1, x=2.0, products=40),
        # a mid-sized target, one incident direction, both polarizations
        _case("solve", "solve_sphere64", nx=64, ny=64, nz=64, m_re=1.5, m_im=0.02, x=5.0),
        # orientation average: 32 directions, both polarizations, one target
        _case("solve", "solve_sweep", nx=96, ny=64, nz=32, m_im=0.05, x=8.0, R=64, products=46),
        # all in 64 bits: a full block of two materials
        _case("solve", "solve_fp64", shape="block", nx=48, ny=48, nz=24, m_re=1.7, m_im=0.3, x=4.0, R=1, prec="fp64",
              materials="two", products=80),
        # a strongly absorbing brick of tilted biaxial crystal, with the guide's other solver
        _case("solve", "solve_brick", shape="block", nx=32, ny=64, nz=64, m_re=0.9656, m_im=1.8628, x=6.187,
              solver="bicgstab2", materials="aniso", products=130),
        # an optimization step: Q_abs forward, its gradient with respect to every dipole's eps backward
        _case("gradient", "gradient_step", nx=32, ny=32, nz=32, m_re=1.4, m_im=0.05, x=2.0, R=1, tol=1e-8, products=110),
        # scattered amplitudes of eight orientations in twelve scattering planes, one degree apart
        _case("farfield", "scattering_planes", nx=96, ny=64, nz=32, m_im=0.05, x=8.0, R=16, thetas=181, planes=12),
        # fields in and around a target, the box extended by half on every side
        _case("nearfield", "near_field", nx=48, ny=48, nz=48, x=3.0, R=2, ext=0.5),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _sides(rng, lo, hi, most):
    while True:
        n = [int(round(_log(rng, lo, hi))) for _ in range(3)]
        if n[0] * n[1] * n[2] <= most:
            return dict(zip(("nx", "ny", "nz"), n))


def draw(rng):
    """One more case: lattices of 8 to 128 sites a side, odd and unequal ones
    among them, 1 to 48 right-hand sides, every precision, solver and kind of
    material; refractive indices that the guide's programs converge for."""
    kind = rng.choice(["matvec", "matvec", "matvec", "solve", "solve", "solve", "spectrum", "gradient", "farfield",
                       "nearfield"])
    c = {"m_re": round(rng.uniform(1.2, 1.6), 3), "m_im": round(_log(rng, 0.003, 0.2), 4)}
    kd = rng.uniform(0.1, 0.25)
    if kind == "matvec":
        c["prec"] = rng.choice(["fp32", "fp32", "df64", "fp64"])
        c.update(_sides(rng, 8, 128, 1 << 20))
        c["R"] = int(round(_log(rng, 1, 16)))
        c["materials"] = rng.choice(["one", "one", "two", "aniso"])
    elif kind == "solve":
        c["prec"] = rng.choice(["refined", "refined", "refined", "fp64"])
        small = c["prec"] == "fp64"
        c.update(_sides(rng, 10, 40 if small else 80, 30000 if small else 250000))
        c["R"] = int(round(_log(rng, 1, 4 if small else 48)))
        c["materials"] = rng.choice(["one", "one", "two", "aniso"])
        c["solver"] = rng.choice(["bicgstab", "bicgstab", "bicgstab2", "qmr"])
    elif kind == "spectrum":
        c.update(_sides(rng, 10, 48, 60000), R=rng.choice([1, 2, 4]), products=40)
    elif kind == "gradient":
        c.update(_sides(rng, 8, 40, 40000), R=1, tol=1e-8, products=110)
    elif kind == "farfield":
        c["prec"] = rng.choice(["refined", "refined", "fp64"])
        c.update(_sides(rng, 10, 96, 200000), R=2 * rng.randint(1, 8), thetas=rng.randint(37, 181),
                 planes=rng.randint(2, 8 if c["prec"] == "refined" else 2))
    else:
        c["prec"] = rng.choice(["refined", "refined", "fp64"])
        c.update(_sides(rng, 10, 40, 40000), R=rng.randint(1, 3), ext=round(rng.uniform(0.2, 0.6), 2))
    c["shape"] = rng.choice(["ellipsoid", "ellipsoid", "block"])
    size = _case(kind, **c)
    c["x"] = round(kd * (3.0 * int(np.count_nonzero(_grid(size))) / (4.0 * math.pi)) ** (1.0 / 3.0), 3)
    return _case(kind, **c)


# ------------------------------------------------------------------ inputs --
def _grid(c):
    """Composition codes [nz, ny, nx]: a full block or the ellipsoid that fills the box."""
    shape = (c["nz"], c["ny"], c["nx"])
    if c["shape"] == "block":
        g = np.ones(shape, np.uint8)
    else:
        z, y, x = [((np.arange(n) - (n - 1) / 2.0) / n) ** 2 for n in shape]
        g = (z[:, None, None] + y[None, :, None] + x[None, None, :] <= 0.25).astype(np.uint8)
    if c["materials"] == "two":
        u = np.random.default_rng(20120514).random(shape)
        g[(u < 0.5) & (g > 0)] = 2
    return g


def _waves(c, seed):
    """R incident waves: random directions, each with both linear polarizations."""
    rng = np.random.default_rng(seed)
    n = (c["R"] + 1) // 2
    z, phi = rng.uniform(-1, 1, n), rng.uniform(0, 2 * np.pi, n)
    s = np.sqrt(1 - z * z)
    k = np.stack([s * np.cos(phi), s * np.sin(phi), z], 1)
    e1 = np.cross([0.0, 0.0, 1.0], k)
    e1 /= np.linalg.norm(e1, axis=1)[:, None]
    e = np.stack([e1, np.cross(k, e1)], 1).reshape(-1, 3)
    return np.repeat(k, 2, 0)[: c["R"]].copy(), e[: c["R"]].astype(np.complex128)


def _index(c, seed):
    """The target's refractive index (the wavelength of a spectrum changes it)."""
    shift = 1.0 + 0.01 * np.random.default_rng(seed + 77).uniform(-1, 1)
    return complex(1.0 + (c["m_re"] - 1.0) * shift, c["m_im"] * shift)


def _indices(c, seed):
    m = _index(c, seed)
    return [m, 1.2 + 0.01j] if c["materials"] == "two" else [m]


AXES = (1.0, 1.05, 0.95)       # principal indices of the biaxial crystal, relative to m
ANGLES = (0.4, 1.1, -0.6)      # its dielectric frame


def _set_materials(ctx, c, seed):
    if c["materials"] == "aniso":
        m = _index(c, seed)
        ctx.set_anisotropic_materials([[m * a for a in AXES]], [ANGLES])
    else:
        ctx.set_materials(_indices(c, seed))


def _site_eps(c, seed, n):
    """Per-dipole dielectric function of an optimization: the index with one per cent of spread."""
    rng = np.random.default_rng(seed + 5)
    return _index(c, seed) ** 2 * (1.0 + 0.01 * rng.standard_normal(n))


def _directions(c):
    theta = np.repeat(np.linspace(0.0, np.pi, c["thetas"])[None], c["planes"], 0).ravel()
    phi = np.repeat(2 * np.pi * np.arange(c["planes"]) / c["planes"], c["thetas"])
    return theta, phi


def _vector(seed, shape, dtype):
    g = torch.Generator(device="cuda").manual_seed(int(seed) + 11)
    return torch.randn(shape, dtype=dtype, device="cuda", generator=g)


def prepare(case, seed):
    c, grid = case, _grid(case)
    k, e = _waves(c, seed)
    n = int(np.count_nonzero(grid))
    st = {"case": c, "k": k, "e": e}
    if c["kind"] == "gradient":
        st["target"] = DipoleTarget(grid, c["x"], k[0], e[0], precision=PREC[c["prec"]], tol=c["tol"])
        st["eps"] = torch.from_numpy(_site_eps(c, seed, n)).cuda()
        return st
    ctx = st["ctx"] = dda.Context(0)
    ctx.set_target(grid)
    _set_materials(ctx, c, seed)
    prec = PREC["fp64"] if c["prec"] == "fp64" else PREC["refined"]
    ctx.prepare_size_parameter(c["x"], prec)
    if c["kind"] == "matvec":
        dtype = torch.complex64 if c["prec"] == "fp32" else torch.complex128
        st["in"] = _vector(seed, (c["R"], 3, n), dtype)
        st["out"] = torch.empty_like(st["in"])
    elif c["kind"] in ("solve", "spectrum"):
        st["out"] = torch.empty((c["R"], 3, n), dtype=torch.complex128, device="cuda")
        st["m"] = _indices(c, seed)
    else:
        st["P"] = _vector(seed, (c["R"], 3, n), torch.complex128).cpu().numpy()
        if c["kind"] == "farfield":
            st["theta"], st["phi"] = _directions(c)
    return st


def _kept(v, c):
    if c["prec"] == "fp64":
        return v
    return v.to(torch.complex64) if isinstance(v, torch.Tensor) else v.astype(np.complex64)


def run(st):
    c = st["case"]
    prec = PREC[c["prec"]]
    if c["kind"] == "matvec":
        dda.dda_matvec_device(st["ctx"].handle, prec, st["k"], st["e"], st["in"], st["out"])
        return st["out"]
    if c["kind"] in ("solve", "spectrum"):
        if c["kind"] == "spectrum":
            st["ctx"].set_materials(st["m"])
            st["ctx"].prepare_size_parameter(c["x"], prec)
        res, _ = dda.dda_solve_device(st["ctx"].handle, prec, st["k"], st["e"], st["out"], tol=c["tol"], maxit=2000,
                                      solver=c["solver"])
        q = np.array([[r["qext"], r["qabs"], r["qsca"]] for r in res])
        return {"P": _kept(st["out"], c), "q": q if c["prec"] == "fp64" else q.astype(np.float32)}
    if c["kind"] == "gradient":
        eps = st["eps"].detach().requires_grad_(True)
        q = QabsFn.apply(eps, st["target"])
        q.backward()
        return {"q": q.detach().to(torch.float32), "grad": _kept(eps.grad, c)}
    if c["kind"] == "farfield":
        return _kept(st["ctx"].farfield(prec, st["k"], st["P"], st["theta"], st["phi"]), c)
    inc, sca, _, _ = st["ctx"].nearfield(prec, st["k"], st["e"], st["P"], [c["ext"]] * 6)
    return {"inc": inc, "sca": _kept(sca, c)}


# -------------------------------------------------------------------- work --
def _product_flops(n):
    """Pruned FFT convolution on the lattice n = (nx, ny, nz), one right-hand side."""
    f = lambda m: 5.0 * 2 * m * math.log2(2 * m)  # noqa: E731
    x, y, z = n
    return 2 * 3 * (y * z * f(x) + z * 2 * x * f(y) + 4 * x * y * f(z)) + 66 * 8.0 * x * y * z


def work(case):
    c = case
    n, lat = int(np.count_nonzero(_grid(c))), (c["nx"], c["ny"], c["nz"])
    s = 8 if c["prec"] in ("fp32", "refined") else 16
    R, green = c["R"], 6.0 * (c["nx"] + 1) * (c["ny"] + 1) * (c["nz"] + 1)
    product = {"bytes": 2.0 * R * 3 * n * s + green * s + 4.0 * n, "flops": R * _product_flops(lat)}
    if c["kind"] == "matvec":
        return product
    if c["kind"] in ("solve", "spectrum", "gradient"):
        return {"bytes": c["products"] * product["bytes"], "flops": c["products"] * product["flops"]}
    if c["kind"] == "farfield":
        nd = c["thetas"] * c["planes"]
        return {"bytes": R * 3 * 16.0 * (n + nd), "flops": 24.0 * R * n * nd}
    box = [v + 2 * math.floor(c["ext"] * v + 0.5) for v in lat]
    ne = box[0] * box[1] * box[2]
    return {"bytes": 16.0 * R * 3 * (n + 2 * ne) + 6 * 16.0 * ne, "flops": R * _product_flops(box)}


# ------------------------------------------------------------------- exact --
class _Lattice:
    """A target's interaction matrix by zero-padded FFTs, complex128 in torch."""

    def __init__(self, grid, kd, box=None, off=(0, 0, 0)):
        dev = "cuda"
        self.kd = kd
        self.n = box or grid.shape[::-1]                       # output box (x, y, z)
        nx, ny, nz = self.n
        self.L = (2 * nz, 2 * ny, 2 * nx)
        occ = np.zeros((nz, ny, nx), np.uint8)
        occ[off[2]: off[2] + grid.shape[0], off[1]: off[1] + grid.shape[1], off[0]: off[0] + grid.shape[2]] = grid
        self.sites = torch.from_numpy(np.flatnonzero(occ)).to(dev)
        self.codes = torch.from_numpy(occ.ravel()[np.flatnonzero(occ)].astype(np.int64)).to(dev)
        d = [torch.fft.fftfreq(m, 1.0 / m, device=dev, dtype=torch.float64) for m in self.L]
        dz, dy, dx = torch.meshgrid(*d, indexing="ij")
        keep = (dx.abs() < nx) & (dy.abs() < ny) & (dz.abs() < nz) & ((dx != 0) | (dy != 0) | (dz != 0))
        r = torch.sqrt(dx * dx + dy * dy + dz * dz)
        r[0, 0, 0] = 1.0
        ph = torch.polar(1.0 / r, kd * r) * keep
        b = torch.complex(-1.0 / (r * r), kd / r)
        u = [dx / r, dy / r, dz / r]
        self.g = {}
        for i in range(3):
            for j in range(i, 3):
                t = u[i] * u[j]
                one = 1.0 if i == j else 0.0
                self.g[i, j] = torch.fft.fftn(ph * (kd * kd * (t - one) + b * (3.0 * t - one)))

    def offdiagonal(self, P, everywhere=False):
        """sum_{l != j} A_jl P_l for one right-hand side P [3, N], at the sites or in the whole box."""
        nx, ny, nz = self.n
        spec = []
        for a in range(3):
            v = torch.zeros(nz * ny * nx, dtype=torch.complex128, device=P.device)
            v[self.sites] = P[a]
            spec.append(torch.fft.fftn(v.view(nz, ny, nx), s=self.L))
        out = []
        for a in range(3):
            y = sum(self.g[min(a, b), max(a, b)] * spec[b] for b in range(3))
            y = torch.fft.ifftn(y)[:nz, :ny, :nx].reshape(-1)
            out.append(y if everywhere else y[self.sites])
        return torch.stack(out)

    def incident(self, k, e, box_centre=None, points=None):
        nx, ny, nz = self.n
        p = self.sites if points is None else points
        cx, cy, cz = box_centre or ((nx - 1) / 2.0, (ny - 1) / 2.0, (nz - 1) / 2.0)
        x, y, z = (p % nx).double() - cx, (p // nx % ny).double() - cy, (p // (nx * ny)).double() - cz
        phase = self.kd * (k[0] * x + k[1] * y + k[2] * z)
        return torch.from_numpy(e).to(p.device)[:, None] * torch.polar(torch.ones_like(phase), phase)[None]


def _inverse_alpha(eps, kd, k, e):
    """Lattice dispersion relation (Draine & Goodman 1993) and its derivative."""
    b1, b2, b3 = -1.8915316, 0.1648469, -1.7700004
    s = float(np.sum(k ** 2 * np.abs(e) ** 2))
    v = 4 * np.pi / 3 * (eps + 2) / (eps - 1) + (b1 + b2 * eps + b3 * eps * s) * kd ** 2 - 2j / 3 * kd ** 3
    return v, -4 * np.pi / (eps - 1) ** 2 + (b2 + b3 * s) * kd ** 2


def _dielectric_axes():
    (ct, cp, cb), (st, sp, sb) = np.cos(ANGLES), np.sin(ANGLES)
    return np.array([[ct, st * cp, st * sp], [-st * cb, ct * cb * cp - sb * sp, ct * cb * sp + sb * cp],
                     [st * sb, -(ct * sb * cp + cb * sp), -(ct * sb * sp - cb * cp)]])


def _diagonal(c, seed, kd, k, e, codes):
    """1/alpha at the sites: [3, 3, N] for tilted crystals, else [N]."""
    if c["materials"] == "aniso":
        ax = _dielectric_axes()
        b = np.array([_inverse_alpha((_index(c, seed) * a) ** 2, kd, k, e)[0] for a in AXES])
        t = torch.from_numpy(np.einsum("j,ja,jb->ab", b, ax, ax)).cuda()
        return t[:, :, None].expand(3, 3, codes.numel())
    b = np.array([_inverse_alpha(m ** 2, kd, k, e)[0] for m in _indices(c, seed)])
    return torch.from_numpy(b).cuda()[codes - 1]


def _apply(lat, beta, x):
    d = (beta * x[None]).sum(1) if beta.dim() == 3 else beta * x
    return lat.offdiagonal(x) + d


def _bicgstab(lat, beta, b, tol=1e-10, most=1500):
    dot = lambda u, v: torch.vdot(u.reshape(-1), v.reshape(-1))  # noqa: E731
    x = torch.zeros_like(b)
    bn = float(torch.linalg.vector_norm(b))
    for _ in range(4):                      # restarts from the true residual
        r = b - _apply(lat, beta, x)
        if float(torch.linalg.vector_norm(r)) <= tol * bn:
            break
        rh, p, v = r.clone(), torch.zeros_like(r), torch.zeros_like(r)
        rho = alpha = omega = torch.ones((), dtype=b.dtype, device=b.device)
        for _ in range(most):
            rho1 = dot(rh, r)
            p = r + (rho1 / rho) * (alpha / omega) * (p - omega * v)
            rho = rho1
            v = _apply(lat, beta, p)
            alpha = rho / dot(rh, v)
            s = r - alpha * v
            t = _apply(lat, beta, s)
            omega = dot(t, s) / dot(t, t)
            x = x + alpha * p + omega * s
            r = s - omega * t
            if float(torch.linalg.vector_norm(r)) <= 0.5 * tol * bn:
                break
    return x


def exact(case, seed):
    c, grid = case, _grid(case)
    k, e = _waves(c, seed)
    n = int(np.count_nonzero(grid))
    aeff = (3.0 * n / (4.0 * math.pi)) ** (1.0 / 3.0)
    kd = c["x"] / aeff
    if c["kind"] == "farfield":
        return _exact_farfield(c, seed, grid, k, kd, n)
    if c["kind"] == "nearfield":
        return _exact_nearfield(c, seed, grid, k, e, kd, n)
    lat = _Lattice(grid, kd)
    if c["kind"] == "gradient":
        eps = _site_eps(c, seed, n)
        beta, dbeta = [torch.from_numpy(v).cuda() for v in _inverse_alpha(eps, kd, k[0], e[0])]
        w = -beta.imag - 2.0 / 3.0 * kd ** 3
        P = _bicgstab(lat, beta, lat.incident(k[0], e[0]))
        nu = _bicgstab(lat, beta, w * P.conj())
        scale = 4.0 * kd / aeff ** 2
        p2, cross = (P.abs() ** 2).sum(0), (nu * P).sum(0) * dbeta
        return {"q": scale * (w * p2).sum(),
                "grad": scale * torch.complex(-dbeta.imag * p2 - 2 * cross.real, -dbeta.real * p2 + 2 * cross.imag)}
    P, Q = [], []
    x = None
    if c["kind"] == "matvec":
        x = _vector(seed, (c["R"], 3, n), torch.complex64 if c["prec"] == "fp32" else torch.complex128)
    for r in range(c["R"]):
        beta = _diagonal(c, seed, kd, k[r], e[r], lat.codes)
        if x is not None:
            P.append(_apply(lat, beta, x[r].to(torch.complex128)))
            continue
        E = lat.incident(k[r], e[r])
        P.append(_bicgstab(lat, beta, E))
        bp = (beta * P[-1][None]).sum(1) if beta.dim() == 3 else beta * P[-1]
        scale = 4.0 * kd / aeff ** 2
        ext = scale * float((E.conj() * P[-1]).imag.sum())
        # P . (1/alpha)^* P^*, less the radiated part
        absorbed = scale * float((P[-1] * bp.conj()).imag.sum() - 2.0 / 3.0 * kd ** 3 * (P[-1].abs() ** 2).sum())
        Q.append([ext, absorbed, ext - absorbed])
    P = torch.stack(P)
    return P if x is not None else {"P": P, "q": np.array(Q)}


def _exact_farfield(c, seed, grid, k, kd, n):
    P = _vector(seed, (c["R"], 3, n), torch.complex128)
    theta, phi = _directions(c)
    nz, ny, nx = grid.shape
    sites = torch.from_numpy(np.flatnonzero(grid)).cuda()
    xyz = torch.stack([sites % nx - (nx - 1) / 2.0, sites // nx % ny - (ny - 1) / 2.0, sites // (nx * ny) - (nz - 1) / 2.0])
    out = []
    for r in range(c["R"]):
        y = np.cross([0.0, 0.0, 1.0], k[r])
        y = y / np.linalg.norm(y)
        z = np.cross(k[r], y)
        d = torch.from_numpy(np.outer(np.cos(theta), k[r]) + np.outer(np.sin(theta) * np.cos(phi), y)
                             + np.outer(np.sin(theta) * np.sin(phi), z)).cuda()
        f = torch.zeros((d.shape[0], 3), dtype=torch.complex128, device="cuda")
        for j in range(0, n, 16384):        # axis by axis: the phases of a lattice separate
            ph = [torch.polar(torch.ones((), dtype=torch.float64, device="cuda").expand(d.shape[0], m),
                              -kd * d[:, a: a + 1] * (torch.arange(m, device="cuda") - (m - 1) / 2.0))
                  for a, m in enumerate((nx, ny, nz))]
            at = [(xyz[a, j: j + 16384] + (m - 1) / 2.0).long() for a, m in enumerate((nx, ny, nz))]
            f += (ph[0][:, at[0]] * ph[1][:, at[1]] * ph[2][:, at[2]]) @ P[r, :, j: j + 16384].T
        dc = d.to(torch.complex128)
        out.append(kd ** 2 * (f - dc * (dc * f).sum(1, keepdim=True)))
    return torch.stack(out)


def _exact_nearfield(c, seed, grid, k, e, kd, n):
    P = _vector(seed, (c["R"], 3, n), torch.complex128)
    own = grid.shape[::-1]
    add = [math.floor(c["ext"] * v + 0.5) for v in own]
    box = tuple(v + 2 * a for v, a in zip(own, add))
    lat = _Lattice(grid, kd, box, add)
    points = torch.arange(box[0] * box[1] * box[2], device="cuda")
    inc = torch.stack([lat.incident(k[r], e[r], points=points) for r in range(c["R"])])
    return {"inc": inc, "sca": torch.stack([-lat.offdiagonal(P[r], True) for r in range(c["R"])])}
