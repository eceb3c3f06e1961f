"""The work that users of this library have it do, as measurable cases.

Every case goes through the package's public entry points (`DeviceProblem`, `DeviceProblem3D`,
`UnevenBatch`, `misfit`) on seeded synthetic models of the kinds `inputs.py` describes: layered VTI
or isotropic media with Gaussian anomalies. A 2D grid of nz x nx cells is zero-padded to the
FFT lengths the input recipes choose (powers of two, and 768 in complex64).

`exact` restates each case in FP64 with plain torch operations on the same (rounded) inputs.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2402_02116_gb300 import dbi, inputs
from paper_2402_02116_gb300.group import UnevenBatch
from paper_2402_02116_gb300.misfit import MisfitProblem, misfit
from paper_2402_02116_gb300.problem import DeviceProblem, DeviceProblem3D

DEV = "cuda"
SCALE = 1e-10  # metres: the size of a wavefield of a unit force


def _case(name, kind, nz, nx, h, src, f_lo, f_hi, nf, amp=0.15, vti=True, c128=False, tol=1e-6):
    return {"name": name, "kind": kind, "nz": nz, "nx": nx, "h": h, "src": src, "f_lo": f_lo, "f_hi": f_hi,
            "nf": nf, "amp": amp, "vti": vti, "c128": c128, "tol": tol}


def listed():
    return [
        # the plain method on a tiny grid: one source, one frequency, double precision; launches
        # and host round trips are all there is
        _case("solve_32_c128", "solve", 32, 32, 10.0, 1, 10.0, 10.0, 1, amp=0.1, vti=False, c128=True, tol=1e-8),
        # the background solve inside the inversion loop at the size of the paper's 2D reservoir
        # example: ragged 45 x 180 cells, 45 sources, one frequency at a time
        _case("solve_45x180", "solve", 45, 180, 20.0, 45, 9.0, 9.0, 1, amp=0.1),
        # the operator on the batched forward workload (32 sources x 8 frequencies)
        _case("apply_256", "apply", 256, 256, 5.0, 32, 5.0, 20.0, 8),
        # a 384-cell member of the uneven workload on FFT length 768
        _case("apply_384", "apply", 384, 384, 5.0, 16, 2.0, 25.0, 6),
        # the operator on the misfit workload, the largest batch: 64 sources x 6 frequencies
        _case("apply_512", "apply", 512, 512, 5.0, 64, 3.0, 18.0, 6),
        # the plain double-precision operator on the linear-step workload (checks, references)
        _case("apply_128_c128", "apply", 128, 128, 10.0, 16, 4.0, 16.0, 4, vti=False, c128=True),
        # one whole gradient: tables, incident fields, forward solves, misfit, adjoint solves
        _case("gradient_512", "gradient", 512, 512, 5.0, 8, 3.0, 18.0, 4, amp=0.05),
        # the matrix-free linear step: one Frechet and one adjoint product for 64 wavefields
        _case("products_128", "products", 128, 128, 10.0, 16, 4.0, 16.0, 4, amp=0.1, vti=False),
        # the paper's own Krylov method, GMRES(30), on wavefields of the forward workload
        _case("gmres_256", "gmres", 256, 256, 5.0, 8, 5.0, 20.0, 8, amp=0.08),
        # grids of 64 to 512 cells in one persistent launch per stage
        {"name": "uneven_40", "kind": "uneven", "members": 40, "max_src": 8, "max_f": 4, "layout": 5},
        # the paper-literal operator (differences on the Green's tensor)
        _case("literal_256", "literal", 256, 256, 5.0, 32, 5.0, 20.0, 8),
        # the 3D example: 80 x 40 x 32 cells, GMRES(30) over 16 sources x 4 frequencies
        {"name": "solve_3d", "kind": "solve3d", "nz": 32, "ny": 40, "nx": 80, "h": 25.0, "src": 16, "f_lo": 3.0,
         "f_hi": 9.0, "nf": 4, "tol": 1e-6},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One case of the same kinds: sizes log-uniform over the range (odd ones included), shrunk in
    sources until it costs no more than the listed case of its kind."""
    kind = rng.choice(["apply", "apply", "apply", "solve", "solve", "gradient", "products", "gmres", "uneven",
                       "literal", "solve3d"])
    most = max(_cost(c) for c in listed() if c["kind"] == kind)
    if kind == "solve":  # solves run at the sizes of a gradient's forward half as well
        most = max(_cost(c) for c in listed()) / 4
    if kind == "uneven":
        c = {"kind": kind, "members": rng.randint(4, 40), "max_src": rng.randint(1, 8), "max_f": rng.randint(1, 4),
             "layout": rng.randint(0, 10 ** 6)}
        while _cost(c) > most and c["members"] > 2:
            c["members"] -= 1
        return c
    if kind == "solve3d":
        c = {"kind": kind, "nz": _log_int(rng, 8, 40), "ny": _log_int(rng, 8, 48), "nx": _log_int(rng, 12, 96),
             "h": 25.0, "src": rng.randint(4, 16), "f_lo": 3.0, "f_hi": rng.uniform(4.0, 9.0), "nf": rng.randint(1, 4),
             "tol": 1e-6}
    else:
        hi = 512 if kind in ("apply", "solve", "gradient") else 256
        nz, nx = _log_int(rng, 20, hi), _log_int(rng, 20, hi)
        h = rng.choice([5.0, 10.0])
        f_hi = rng.uniform(4.0, 90.0 / h)
        c128 = kind in ("apply", "solve") and rng.random() < 0.2
        amp = rng.uniform(0.05, 0.15) if kind in ("apply", "literal") else rng.uniform(0.03, 0.06)
        c = _case("", kind, nz, nx, h, rng.randint(4, 64), 3.0, f_hi, rng.randint(2, 8), amp=amp,
                  vti=rng.random() < 0.7, c128=c128)
        del c["name"]
        if c128:
            most = min(most, max(_cost(d) for d in listed() if d.get("c128")))
    while _cost(c) > most and (c["src"] > 1 or c["nf"] > 1):
        key = "src" if c["src"] > 1 else "nf"
        c[key] = max(1, int(c[key] * 0.8))
    return c


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _surface(n, count):
    return inputs.surface_line(n, min(n, count))


def _perturb(rng, shape, count=4, amp=0.15):
    """Three layers and `count` Gaussian anomalies, +/- amp per parameter, on [params][nz][nx]."""
    p, nz, nx = shape
    pert = np.zeros(shape)
    for z0 in np.sort(rng.uniform(0.1 * nz, 0.9 * nz, 3)).astype(int):
        pert[:, z0:, :] = rng.uniform(-amp, amp, p)[:, None, None]
    for _ in range(count):
        cz, cx = rng.uniform(0.2, 0.8, 2) * (nz, nx)
        g = inputs.gaussian_bump(nz, nx, cz, cx, rng.uniform(0.02, 0.08) * max(nz, nx) + 1.0)
        pert += (amp * rng.choice([-1.0, 1.0], p))[:, None, None] * g[None]
    return np.clip(pert, -amp, amp)


def _workload(c, seed):
    rng = np.random.default_rng(seed)
    nz, nx = c["nz"], c["nx"]
    if c["vti"]:
        bg = inputs.vti_background(nz, nx)
        rho0, a0, b0 = inputs.isotropic_reference_for(bg)
    else:
        rho0, a0, b0 = 2000.0, 2000.0, 1155.0
        bg = inputs.isotropic_model(nz, nx, rho0, a0, b0)
    model = bg * (1.0 + _perturb(rng, bg.shape, amp=c["amp"]))
    if not c["c128"]:
        model = model.astype(np.float32).astype(np.float64)
    src = _surface(nx, c["src"])
    rec = np.arange(0, nx, 2)
    lens = [inputs.fft_len(n, radix3=not c["c128"] and c["kind"] != "literal") for n in (nz, nx)]
    return inputs.Workload(
        name="case", nz=nz, nx=nx, h=c["h"], lz=lens[0], lx=lens[1], rho0=rho0, alpha0=a0, beta0=b0, model=model,
        freqs_hz=np.linspace(c["f_lo"], c["f_hi"], c["nf"]), src_cells=np.stack([np.zeros_like(src), src], axis=1),
        src_force=np.tile([0.0, 1.0], (len(src), 1)), rec_cells=np.stack([np.zeros_like(rec), rec], axis=1),
        krylov_tol=c["tol"], seed=seed)


def _members(c, seed):
    """The uneven batch: grids, sources and frequencies from the layout, models from the seed."""
    lay, out = np.random.default_rng(c["layout"]), []
    for k in range(c["members"]):
        n = int(lay.choice([64, 128, 256, 384, 512]))
        d = _case("", "uneven", n, n, 5.0, int(lay.integers(1, c["max_src"] + 1)), 2.0 + float(lay.uniform(0, 3)),
                  float(lay.uniform(6, 25)), int(lay.integers(1, c["max_f"] + 1)), vti=bool(lay.integers(0, 2)))
        out.append((d, _workload(d, seed * 1000 + k) if seed is not None else None))
    return out


def _workload3(c, seed):
    n = [c["nz"], c["ny"], c["nx"]]
    w = inputs.hess3d_like(*n, h=c["h"], n_src=c["src"], freqs=np.linspace(c["f_lo"], c["f_hi"], c["nf"]), seed=seed)
    w.model = w.model.astype(np.float32).astype(np.float64)
    w.krylov_tol = c["tol"]
    return w


def _waves(w, seed, dtype):
    """[B][2][nz][nx] wavefields: plane waves at each problem's P and S wavenumbers, of the size of a
    unit force's response."""
    gen = torch.Generator().manual_seed(seed)
    om = torch.tensor(w.omegas[w.problem_fidx()])[:, None, None]
    k = om / torch.tensor([w.alpha0, w.beta0, w.beta0], dtype=torch.float64)
    B = len(om)
    th = 2 * math.pi * torch.rand(B, 2, 3, generator=gen, dtype=torch.float64)
    amp = SCALE * torch.randn(B, 2, 3, generator=gen, dtype=torch.complex128)
    z, x = (torch.arange(n, dtype=torch.float64, device=DEV) * w.h for n in (w.nz, w.nx))
    kz, kx, amp = ((k * torch.sin(th)).to(DEV), (k * torch.cos(th)).to(DEV), amp.to(DEV))
    ez = (amp[..., None] * torch.exp(-1j * kz[..., None] * z)).to(dtype)
    ex = torch.exp(-1j * kx[..., None] * x).to(dtype)
    u = ez[:, :, 0, :, None] * ex[:, :, 0, None, :]
    for j in (1, 2):
        u += ez[:, :, j, :, None] * ex[:, :, j, None, :]
    return u.contiguous()


def _noise(shape, seed, dtype):
    gen = torch.Generator().manual_seed(seed)
    return torch.randn(shape, generator=gen, dtype=dtype).to(DEV)


def _dm(w, seed, dtype):
    """A model perturbation of up to 5 %."""
    rng = np.random.default_rng(seed + 1)
    ref = w.model.mean(axis=(1, 2))[:, None, None]
    return torch.tensor(0.3 * ref * _perturb(rng, w.model.shape, amp=0.15)).to(DEV, dtype)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "uneven":
        ws = [w for _, w in _members(case, seed)]
        problems = [DeviceProblem(w, dbi.C64, with_space=False) for w in ws]
        batch = UnevenBatch(problems)
        batch.bind(dbi.OP_APPLY)
        u = batch.join([_waves(w, seed + k, torch.complex64) for k, w in enumerate(ws)])
        return {"kind": kind, "batch": batch, "u": u}
    if kind == "solve3d":
        P = DeviceProblem3D(_workload3(case, seed), dbi.C64)
        return {"kind": kind, "P": P}
    prec = dbi.C128 if case["c128"] else dbi.C64
    w = _workload(case, seed)
    P = DeviceProblem(w, prec)
    s = {"kind": kind, "P": P}
    nrec = len(w.rec_cells)
    if kind in ("apply", "literal", "products"):
        s["u"] = _waves(w, seed, P.cdt)
    if kind == "literal":
        P.Dhat  # tabulated on first use, once per problem
    if kind in ("products", "gradient"):
        s["r"] = (SCALE * _noise((P.B, nrec, 2), seed, torch.complex128)).to(P.cdt)
    if kind == "products":
        s["dm"] = _dm(w, seed, P.rdt)
    return s


def run(state):
    kind = state["kind"]
    if kind == "uneven":
        return state["batch"].apply(state["u"])
    P = state["P"]
    if kind == "apply":
        return P.apply(state["u"])
    if kind == "literal":
        return P.apply_k(state["u"])
    if kind in ("solve", "solve3d"):
        u, _, _, code = P.solve(P.incident())
        return [u, code]
    if kind == "gmres":
        u, _, _, code = P.solve_gmres(P.incident())
        return [u, code]
    if kind == "products":
        return [P.frechet(state["u"], state["dm"]), P.adjoint(state["u"], state["r"])]
    # gradient: the tables of the model's frequencies, then the differentiable misfit
    P.Ghat, P.Gspace = dbi.greens_tabulate(P.grid, P.ref, P.omega, P.precision)
    m = P.m.clone().requires_grad_(True)
    phi = misfit(m, MisfitProblem(P, state["r"], tol=P.w.krylov_tol))
    phi.backward()
    return {"phi": phi.detach().to(P.rdt), "grad": m.grad}


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
ITERATIONS = 20  # BiCGSTAB iterations of a solve to 1e-6 on these models (two operator passes each)


def _pass_flops(c):
    """5 L log2 L per transform over the non-zero rows and all columns, forward and inverse, and the
    product with the symmetric kernel, for one problem."""
    f = lambda L: 5.0 * L * math.log2(L)  # noqa: E731
    if c["kind"] == "solve3d":
        lz, ly, lx = (inputs.fft_len(c[k]) for k in ("nz", "ny", "nx"))
        return 6 * (c["nz"] * c["ny"] * f(lx) + c["nz"] * lx * f(ly) + lx * ly * f(lz)) + 66 * lx * ly * lz
    lz, lx = (inputs.fft_len(c[k], radix3=not c["c128"] and c["kind"] != "literal") for k in ("nz", "nx"))
    n_in, n_out, mul = (5, 2, 80) if c["kind"] == "literal" else (2, 2, 28)
    return (n_in + n_out) * (c["nz"] * f(lx) + lx * f(lz)) + mul * lz * lx


def _shape(c):
    """(problems, cells, FFT points, components, parameters)"""
    if c["kind"] == "solve3d":
        k = int(round(math.sqrt(c["src"])))
        n_src = min(c["src"], k * max(1, c["src"] // k))
        pts = math.prod(inputs.fft_len(c[k]) for k in ("nz", "ny", "nx"))
        return n_src * c["nf"], c["nz"] * c["ny"] * c["nx"], pts, 3, 6
    pts = math.prod(inputs.fft_len(c[k], radix3=not c["c128"] and c["kind"] != "literal") for k in ("nz", "nx"))
    return min(c["src"], c["nx"]) * c["nf"], c["nz"] * c["nx"], pts, 2, 5


def _passes(c):
    return {"apply": 1, "literal": 1, "uneven": 1, "solve": 2 * ITERATIONS, "gmres": 30, "solve3d": 15,
            "gradient": 4 * ITERATIONS + 1, "products": 4 * ITERATIONS + 2}[c["kind"]]


def _cost(c):
    if c["kind"] == "uneven":
        return sum(_cost(dict(d, kind="apply")) for d, _ in _members(c, None))
    return _shape(c)[0] * _pass_flops(c) * _passes(c) * (30.0 if c.get("c128") else 1.0)


def work(case):
    if case["kind"] == "uneven":
        parts = [work(dict(d, kind="apply")) for d, _ in _members(case, None)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    B, cells, pts, comps, params = _shape(case)
    size = 16 if case.get("c128") else 8
    field = B * comps * cells * size
    model = params * cells * size // 2
    tables = case["nf"] * pts * (6 if comps == 3 else 3) * size
    bytes_ = {"apply": 2 * field + model + tables, "literal": 2 * field + model + 3 * tables,
              # a solve reads the tables and writes the wavefields; its right-hand side is made in the pass
              "solve": field + model + 2 * tables, "gmres": field + model + 2 * tables,
              "solve3d": field + model + 2 * tables,
              "gradient": 2 * model, "products": field + 3 * model + tables}[case["kind"]]
    return {"bytes": float(bytes_), "flops": float(B * _pass_flops(case) * _passes(case))}


# ---------------------------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------------------------
def _diff(v, axis, h):
    """Central difference along `axis` of the trailing grid axes, zero outside the grid."""
    n = v.shape[axis]
    out = torch.zeros_like(v)
    if n > 1:
        out.narrow(axis, 0, n - 1).add_(v.narrow(axis, 1, n - 1))
        out.narrow(axis, 1, n - 1).sub_(v.narrow(axis, 0, n - 1))
    return out.div_(2.0 * h)


def _cplx(re, im):
    return torch.complex(re, im)


def _hankel01(z):
    """H0 and H1 of the second kind. Up to z = 2 from torch's Bessel functions; above, where those
    lose digits, from H_n^(1)(z) = sqrt(2 / (pi z)) e^{i (z - n pi/2 - pi/4)} / Gamma(n + 1/2)
    times the integral over the real line of e^{-s^2} s^{2n} (1 + i s^2 / 2z)^{n - 1/2} (Hankel's
    integral with u = s^2), which the trapezoidal rule takes to rounding."""
    sp = torch.special
    zs, zl = z.clamp(max=2.0), z.clamp(min=2.0)
    small = _cplx(sp.bessel_j0(zs), -sp.bessel_y0(zs)), _cplx(sp.bessel_j1(zs), -sp.bessel_y1(zs))
    step, i0, i1 = 0.25, 1.0, 0.0
    for n in range(1, 26):
        s2 = (n * step) ** 2
        root = torch.sqrt(_cplx(torch.ones_like(zl), s2 / (2.0 * zl)))
        i0 = i0 + 2.0 * math.exp(-s2) / root
        i1 = i1 + 2.0 * math.exp(-s2) * s2 * root
    pre = torch.sqrt(2.0 / (math.pi * zl)) * torch.exp(1j * (zl - math.pi / 4)) * (step / math.sqrt(math.pi))
    large = (pre * i0).conj(), (pre * (-2j) * i1).conj()
    return tuple(torch.where(z < 2.0, a, b) for a, b in zip(small, large))


def _lattice2(w, om, nz, nx):
    """G11, G13, G33 on the offsets |dz| < nz, |dx| < nx, [3][2nz-1][2nx-1]."""
    y3 = torch.arange(-(nz - 1), nz, dtype=torch.float64, device=DEV)[:, None] * w.h
    y1 = torch.arange(-(nx - 1), nx, dtype=torch.float64, device=DEV)[None, :] * w.h
    r = torch.sqrt(y1 * y1 + y3 * y3)
    r[nz - 1, nx - 1] = w.h
    A, B, self_ = 0, 0, 0
    a = w.h / math.sqrt(math.pi)
    for vel, sign in ((w.alpha0, 1.0), (w.beta0, -1.0)):
        z = om * r / vel
        h0, h1 = _hankel01(z)
        A = A + h0 / vel ** 2
        B = B + sign * (2.0 * h1 / z - h0) / vel ** 2
        ka = om * a / vel
        h1a = complex(_hankel01(torch.tensor([ka], dtype=torch.float64))[1].item())
        self_ += (2.0 * h1a / ka - 4j / (math.pi * ka * ka)) / vel ** 2
    pre = 1.0 / (8j * w.rho0)
    c1, c3 = y1 / r, y3 / r
    G = torch.stack([pre * (A - B * (2 * c1 * c1 - 1)), pre * (-B * 2 * c1 * c3), pre * (A - B * (2 * c3 * c3 - 1))])
    G[:, nz - 1, nx - 1] = torch.tensor([pre * self_, 0.0, pre * self_], dtype=torch.complex128, device=DEV)
    return G


def _lattice3(w, om):
    n = (w.nz, w.ny, w.nx)
    y = [torch.arange(-(m - 1), m, dtype=torch.float64, device=DEV) * w.h for m in n]
    Z, Y, X = torch.meshgrid(*y, indexing="ij")
    r = torch.sqrt(X * X + Y * Y + Z * Z)
    o = (w.nz - 1, w.ny - 1, w.nx - 1)
    r[o] = w.h
    g = (X / r, Y / r, Z / r)
    terms = []
    for vel in (w.alpha0, w.beta0):
        k = om / vel
        D = torch.exp(-1j * k * r) / (4 * math.pi * w.rho0 * vel * vel * r)
        q = 1.0 / (1j * k * r)
        terms.append((D, q + q * q))
    (Dp, Qp), (Ds, Qs) = terms
    a = w.h * (3.0 / (4.0 * math.pi)) ** (1.0 / 3.0)
    mean = lambda k: 3 * (np.exp(-1j * k * a) * (1 + 1j * k * a) - 1) / (4 * math.pi * a ** 3 * k * k)  # noqa: E731
    ks, kp = om / w.beta0, om / w.alpha0
    self_ = complex((2 * ks * ks * mean(ks) + kp * kp * mean(kp)) / (3 * w.rho0 * om * om))
    out = []
    for i in range(3):
        for j in range(i, 3):
            gg, d = g[i] * g[j], 1.0 if i == j else 0.0
            e = Dp * (gg + (3 * gg - d) * Qp) - Ds * ((gg - d) + (3 * gg - d) * Qs)
            e[o] = self_ if i == j else 0.0
            out.append(e)
    return torch.stack(out)


def _spectrum(lat, lens):
    """FFT of the offsets placed on the periodic grid."""
    dims = list(range(1, lat.ndim))
    E = torch.zeros((lat.shape[0], *lens), dtype=lat.dtype, device=DEV)
    E[tuple([slice(None)] + [slice(0, n) for n in lat.shape[1:]])] = lat
    return torch.fft.fftn(torch.roll(E, [-((n - 1) // 2) for n in lat.shape[1:]], dims), dim=dims)


class _Exact:
    """The discrete problem of a workload in complex128, a batch of problems at a time."""

    def __init__(self, w, literal=False):
        self.w, self.three, self.literal = w, hasattr(w, "ny"), literal
        self.grid = (w.nz, w.ny, w.nx) if self.three else (w.nz, w.nx)
        self.lens = (w.lz, w.ly, w.lx) if self.three else (w.lz, w.lx)
        self.nc = 3 if self.three else 2
        self.om = torch.tensor(w.omegas, device=DEV)
        lat = [_lattice3(w, om) if self.three else _lattice2(w, om, w.nz, w.nx) for om in w.omegas]
        self.lat = torch.stack(lat)
        self.G = torch.stack([_spectrum(v, self.lens) for v in lat])
        if literal:
            ext = [_lattice2(w, om, w.nz + 1, w.nx + 1) for om in w.omegas]
            d1 = [(e[:, 1:-1, 2:] - e[:, 1:-1, :-2]) / (2 * w.h) for e in ext]
            d3 = [(e[:, 2:, 1:-1] - e[:, :-2, 1:-1]) / (2 * w.h) for e in ext]
            self.D = torch.stack([torch.cat([_spectrum(a, self.lens), _spectrum(b, self.lens)])
                                  for a, b in zip(d1, d3)])
        a2, b2 = w.alpha0 ** 2, w.beta0 ** 2
        ref = w.rho0 * np.array([1.0, a2, a2 - 2 * b2, a2, b2, b2])[:6 if self.three else 5]
        self.ref = torch.tensor(ref, device=DEV).reshape(-1, *([1] * len(self.grid)))
        self.dm = torch.tensor(w.model, device=DEV) - self.ref
        self.fidx = torch.tensor(w.problem_fidx(), device=DEV).long()
        self.srcs = w.problem_src()

    def strain(self, u):
        h, d = self.w.h, _diff
        if self.three:
            a = (-1, -2, -3)
            g = lambda c, k: d(u[:, c], a[k], h)  # noqa: E731
            return [g(0, 0), g(1, 1), g(2, 2), g(1, 2) + g(2, 1), g(0, 2) + g(2, 0), g(0, 1) + g(1, 0)]
        return [d(u[:, 0], -1, h), d(u[:, 1], -2, h), d(u[:, 0], -2, h) + d(u[:, 1], -1, h)]

    def stress(self, u, m):
        e = self.strain(u)
        if self.three:
            c12 = m[1] - 2 * m[5]
            return [m[1] * e[0] + c12 * e[1] + m[2] * e[2], c12 * e[0] + m[1] * e[1] + m[2] * e[2],
                    m[2] * (e[0] + e[1]) + m[3] * e[2], m[4] * e[3], m[4] * e[4], m[5] * e[5]]
        return [m[1] * e[0] + m[2] * e[1], m[2] * e[0] + m[3] * e[1], m[4] * e[2]]

    def source(self, u, m, f):
        s, h, d = self.stress(u, m), self.w.h, _diff
        w2 = (self.om[f] ** 2).reshape(-1, *([1] * (u.ndim - 1)))
        if self.three:
            div = [d(s[0], -1, h) + d(s[5], -2, h) + d(s[4], -3, h), d(s[5], -1, h) + d(s[1], -2, h) + d(s[3], -3, h),
                   d(s[4], -1, h) + d(s[3], -2, h) + d(s[2], -3, h)]
        else:
            div = [d(s[0], -1, h) + d(s[2], -2, h), d(s[2], -1, h) + d(s[1], -2, h)]
        return w2 * m[0] * u + torch.stack(div, 1)

    def kernel(self, i, j, f):
        if not self.three:
            return self.G[f, i + j]
        i, j = min(i, j), max(i, j)
        return self.G[f, (0, 3, 5)[i] + j - i]

    def convolve(self, src, f, literal=False):
        dims = list(range(-len(self.grid), 0))
        S = torch.fft.fftn(src, s=self.lens, dim=dims)
        out = []
        for i in range(self.nc):
            if literal:  # sources w^2 drho u1, w^2 drho u3, sigma1, sigma5, sigma3
                D = self.D
                ker = [self.G[f, i], self.G[f, i + 1]] + [D[f, i], D[f, 3 + i] + D[f, 1 + i], D[f, 4 + i]]
            else:
                ker = [self.kernel(i, j, f) for j in range(self.nc)]
            acc = ker[0] * S[:, 0]
            for j in range(1, len(ker)):
                acc += ker[j] * S[:, j]
            out.append(torch.fft.ifftn(acc, dim=dims)[(slice(None),) + tuple(slice(0, n) for n in self.grid)])
        return self.w.h ** len(self.grid) * torch.stack(out, 1)

    def apply(self, u, f):
        if self.literal:
            s = self.stress(u, self.dm)
            w2 = (self.om[f] ** 2).reshape(-1, 1, 1, 1)
            rho = w2 * self.dm[0] * u
            return u - self.convolve(torch.stack([rho[:, 0], rho[:, 1], s[0], s[2], s[1]], 1), f, True)
        return u - self.convolve(self.source(u, self.dm, f), f)

    def incident(self, b):
        """Incident fields of the problems b (a list of indices)."""
        out = []
        for p in b:
            s = self.srcs[p]
            cell, force = self.w.src_cells[s], self.w.src_force[s]
            lat = self.lat[int(self.fidx[p])]
            win = lat[(slice(None),) + tuple(slice(n - 1 - int(c), 2 * n - 1 - int(c))
                                             for n, c in zip(self.grid, cell))]
            if self.three:
                idx = ((0, 1, 2), (1, 3, 4), (2, 4, 5))
            else:
                idx = ((0, 1), (1, 2))
            out.append(torch.stack([sum(float(force[j]) * win[row[j]] for j in range(self.nc)) for row in idx]))
        return torch.stack(out)

    def solve(self, rhs, f, tol=1e-10, most=400):
        """BiCGSTAB over the batch, every problem with its own scalars."""
        dims = list(range(1, rhs.ndim))
        col = lambda v: v.reshape(-1, *([1] * (rhs.ndim - 1)))  # noqa: E731
        dot = lambda a, b: torch.sum(a.conj() * b, dims)  # noqa: E731
        safe = lambda v: torch.where(v == 0, torch.ones_like(v), v)  # noqa: E731
        scale = 1.0 / safe(rhs.abs().amax(dims))
        r = rhs * col(scale)
        x, hat, p, v = torch.zeros_like(r), r.clone(), torch.zeros_like(r), torch.zeros_like(r)
        b2 = dot(r, r).real
        rho = al = om = torch.ones_like(b2, dtype=torch.complex128)
        live = b2 > 0
        for _ in range(most):
            if not bool(live.any()):
                break
            new = dot(hat, r)
            beta = torch.where(live, new / safe(rho) * al / safe(om), 0)
            p = r + col(beta) * (p - col(om) * v)
            v = self.apply(p, f)
            al = torch.where(live, new / safe(dot(hat, v)), 0)
            s = r - col(al) * v
            t = self.apply(s, f)
            om = torch.where(live, dot(t, s) / safe(dot(t, t)), 0)
            x += col(al) * p + col(om) * s
            r = torch.where(col(live), s - col(om) * t, r)
            rho = new
            live = live & (dot(r, r).real > tol * tol * b2)
        return x / col(scale)

    def sample(self, u):
        rec = torch.tensor(self.w.rec_cells, device=DEV)
        return u[:, :, rec[:, 0], rec[:, 1]].transpose(1, 2)

    def adjoint(self, u_b, r, f):
        """Re J^H r: the conjugate residual back-propagated from the receivers, then the imaging."""
        q = torch.zeros_like(u_b)
        rec = torch.tensor(self.w.rec_cells, device=DEV)
        q[:, :, rec[:, 0], rec[:, 1]] = r.conj().transpose(1, 2)
        u_a = self.solve(self.convolve(q, f), f)
        ea, eb = self.strain(u_a), self.strain(u_b)
        w2 = (self.om[f] ** 2).reshape(-1, 1, 1)
        g = [(w2 * (u_a * u_b).sum(1)).real, -(ea[0] * eb[0]).real, -(ea[0] * eb[1] + ea[1] * eb[0]).real,
             -(ea[1] * eb[1]).real, -(ea[2] * eb[2]).real]
        return torch.stack([v.sum(0) for v in g])


def _chunks(n, E):
    """Problems at a time: about 4 GB of one padded complex128 field."""
    step = max(1, int(4e9 / (16 * 5 * math.prod(E.lens))))
    return [list(range(b, min(n, b + step))) for b in range(0, n, step)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "uneven":
        out = []
        for k, (_, w) in enumerate(_members(case, seed)):
            E, u = _Exact(w), _waves(w, seed + k, torch.complex64).to(torch.complex128)
            out += [E.apply(u[c], E.fidx[c]).reshape(-1) for c in _chunks(len(u), E)]
        return torch.cat(out)
    w = _workload3(case, seed) if kind == "solve3d" else _workload(case, seed)
    E = _Exact(w, literal=kind == "literal")
    B = w.n_problems
    if kind in ("apply", "literal"):
        u = _waves(w, seed, torch.complex128 if case["c128"] else torch.complex64)
        return torch.cat([E.apply(u[c].to(torch.complex128), E.fidx[c]) for c in _chunks(B, E)])
    if kind in ("solve", "gmres", "solve3d"):
        return [torch.cat([E.solve(E.incident(c), E.fidx[c]) for c in _chunks(B, E)]), None]
    cdt = torch.complex128 if case["c128"] else torch.complex64
    r = (SCALE * _noise((B, len(w.rec_cells), 2), seed, torch.complex128)).to(cdt).to(torch.complex128)
    if kind == "products":
        u = _waves(w, seed, cdt).to(torch.complex128)
        dm = _dm(w, seed, torch.float64 if case["c128"] else torch.float32).double()
        d, g = [], 0
        for c in _chunks(B, E):
            f = E.fidx[c]
            d.append(E.sample(E.solve(E.convolve(E.source(u[c], dm, f), f), f)))
            g = g + E.adjoint(u[c], r[c], f)
        return [torch.cat(d), g]
    phi, g = 0, 0
    for c in _chunks(B, E):
        f = E.fidx[c]
        u = E.solve(E.incident(c), f)
        res = E.sample(u) - r[c]
        phi = phi + 0.5 * torch.sum(res.abs() ** 2)
        g = g + E.adjoint(u, res, f)
    return {"phi": phi, "grad": g}
