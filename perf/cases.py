"""Performance cases: what a user of this framework has it do, as timed passes.

A pass is one whole solve (or one drained batch of solves) through the public
Python entry points, from the density and the starting potential a program has
in hand to the solution in its own tensor.  The listed cases cover the
grids, stencils, precisions, methods and boundaries that the library's own
configurations, tests and benchmark use, from the smallest serving request to
the 512^3 workloads; draw() gives more of the same ranges.
"""
import math

import numpy as np
import torch

from paper_2605_03563_gb300 import Batch, CartesianSolver, SphericalSolver

DEV = "cuda"
PI4 = 4.0 * math.pi


# ------------------------------------------------------------------ the cases
def _cart(name, n, **kw):
    c = {"kind": "cart", "nx": n[0], "ny": n[1], "nz": n[2], "order": 2, "compact": 0, "method": "mg",
         "prec": "fp64", "nu": 2, "inner": 1, "tol": 1e-10, "bc": "multipole", "lmax": 4, "rho": "blobs",
         "start": "cold", "box": "equal", "omega": 1.0, "schedule": "fixed", "max_iter": 100}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def _sph(name, nr, nt, np_, **kw):
    c = {"kind": "sph", "nr": nr, "nt": nt, "np": np_, "method": "bicgstab", "prec": "fp64", "tol": 1e-8,
         "lmax": 6, "r_in": 0.01, "max_iter": 30000}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def _batch(name, sizes, **kw):
    c = {"kind": "batch", "sizes": " ".join(str(n) for n in sizes), "prec": "mixed_fp32", "inner": 3, "nu": 2,
         "tol": 1e-10, "lmax": 4, "step": 2}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest request of the serving stream, at its looser tolerance
        _cart("mg_fp64_32", (32, 32, 32), tol=1e-6),
        # a mid-size step of a slowly moving density, started from the previous step's potential
        _cart("mg_fp64_96_warm", (96, 96, 96), start="warm"),
        # a ragged box with a different spacing on every axis
        _cart("mg_fp64_box_160_112_208", (160, 112, 208), box="unit"),
        # the headline workload: cold start to 1e-10, FP64 and FP32 refinement (3 inner cycles)
        _cart("mg_fp64_256", (256, 256, 256)),
        _cart("mg_fp32_256", (256, 256, 256), prec="mixed_fp32", inner=3),
        # the fourth-order stencil on a turbulent density: FP64, and at full size with BF16 storage
        _cart("mg13_fp64_192", (192, 192, 192), order=4, lmax=8, rho="lognormal"),
        _cart("mg13_bf16_512", (512, 512, 512), order=4, lmax=8, rho="lognormal", prec="mixed_bf16", inner=2),
        # the sixth-order compact scheme on two spheres, V(3,3) in FP64, V(2,2) in FP32 refinement
        _cart("compact6_fp64_256", (256, 256, 256), compact=6, nu=3, tol=1e-6, rho="spheres"),
        _cart("compact6_fp32_512", (512, 512, 512), compact=6, nu=2, tol=1e-6, rho="spheres", prec="mixed_fp32",
              inner=2),
        # red-black SOR on the uniform sphere with its closed-form boundary values
        _cart("sor_32", (32, 32, 32), method="sor", omega=1.8, bc="dirichlet", rho="ball", max_iter=4000),
        # BiCGSTAB on a graded spherical grid
        _sph("sph_bicgstab_96_48_32", 96, 48, 32),
        # a queue of small requests drained by the batched executor
        _batch("batch_fp32_24", (32, 64, 96, 128, 48, 80) * 4),
    ]


def _mg_size(rng, lo, hi):
    """A multigrid-able interval count b 2^k, b in 8..15, log-uniform in [lo, hi]."""
    for _ in range(200):
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        k = max(1, int(math.floor(math.log2(v / 8.0))))
        n = min(15, max(8, int(round(v / 2 ** k)))) * 2 ** k
        if lo <= n <= hi:
            return n
    return lo


def draw(rng):
    kind = rng.choice(["mg", "mg", "mg", "mg13", "compact", "point", "sph", "batch"])
    tol = rng.choice([1e-6, 1e-8, 1e-10])
    if kind == "mg":
        prec = rng.choice(["fp64", "fp64", "mixed_fp32", "mixed_bf16"])
        n = _mg_size(rng, 32, 288)
        if rng.random() < 0.35:   # a box with other counts on y and z (same number of levels)
            k = int(math.floor(math.log2(n / 8.0)))
            m = [rng.randint(8, 15) * 2 ** k for _ in range(2)]
            return _cart("", (n, m[0], m[1]), prec=prec, inner=rng.choice([1, 2, 3]) if prec != "fp64" else 1,
                         tol=tol, box=rng.choice(["equal", "unit"]), lmax=rng.choice([2, 4, 6]),
                         nu=rng.choice([1, 2]))
        return _cart("", (n, n, n), prec=prec, inner=rng.choice([1, 2, 3]) if prec != "fp64" else 1, tol=tol,
                     lmax=rng.choice([2, 4, 6]), start=rng.choice(["cold", "cold", "warm"]), nu=rng.choice([1, 2]))
    if kind == "mg13":
        prec = rng.choice(["fp64", "mixed_fp32", "mixed_bf16"])
        n = _mg_size(rng, 32, 224 if prec == "fp64" else 320)
        return _cart("", (n, n, n), order=4, rho="lognormal", prec=prec, lmax=rng.choice([4, 8]),
                     inner=rng.choice([1, 2]) if prec != "fp64" else 1, tol=tol, nu=2)
    if kind == "compact":
        prec = rng.choice(["fp64", "mixed_fp32"])
        n = _mg_size(rng, 48, 256 if prec == "fp64" else 384)
        return _cart("", (n, n, n), compact=rng.choice([2, 4, 6]), nu=rng.choice([1, 2, 3]), tol=rng.choice([1e-6, 1e-8]),
                     rho="spheres", prec=prec, inner=2 if prec != "fp64" else 1)
    if kind == "point":   # the single-level methods, on sizes that need not be even
        method = rng.choice(["sor", "cg", "pcg"])
        n = int(round(math.exp(rng.uniform(math.log(24), math.log(80)))))
        return _cart("", (n, n, n), method=method, bc="dirichlet", rho="ball", max_iter=8000,
                     schedule=rng.choice(["chebyshev", "optimal"]) if method == "sor" else "fixed", tol=tol)
    if kind == "sph":
        method = rng.choice(["bicgstab", "sor"])
        nr, nt = rng.randint(40, 110), rng.randint(12, 48)
        return _sph("", nr, nt, 2 * rng.randint(4, 16), method=method, tol=1e-8, lmax=rng.choice([2, 4, 6]))
    sizes = [_mg_size(rng, 32, 128) for _ in range(rng.randint(6, 24))]
    return _batch("", sizes, prec=rng.choice(["fp64", "mixed_fp32"]), inner=rng.choice([1, 2, 3]), tol=tol)


# ------------------------------------------------------------------ inputs
def _box(c):
    if c["box"] == "unit":
        return (0.0, 0.0, 0.0), (1.0, 1.0, 1.0)
    m = max(c["nx"], c["ny"], c["nz"])   # equal spacings, the longest axis of length 1
    # spacing 1/m on every axis: n/m is exact enough for equal spacings when n and m share their powers of two
    return (0.0, 0.0, 0.0), (c["nx"] / m, c["ny"] / m, c["nz"] / m)


def _axes(c):
    """Node coordinates (x, y, z) of the field layout, ghost layers included."""
    g = c["order"] // 2
    lo, hi = _box(c)
    out = []
    for a, n in enumerate((c["nx"], c["ny"], c["nz"])):
        i = torch.arange(-(g - 1), n + g, dtype=torch.float64, device=DEV)
        out.append(lo[a] + i * ((hi[a] - lo[a]) / n))
    return out


def _blobs(c, rng, shift=0.0):
    x, y, z = _axes(c)
    _, hi = _box(c)
    s = min(hi)
    rho = torch.zeros((z.numel(), y.numel(), x.numel()), dtype=torch.float64, device=DEV)
    for _ in range(8):
        u, sig, amp = rng.uniform(0.2, 0.8, 3), s * rng.uniform(0.02, 0.08), rng.uniform(0.5, 2.0)
        e = [torch.exp(-0.5 * ((q - (u[a] * hi[a] + shift * s)) / sig) ** 2) for a, q in enumerate((x, y, z))]
        rho += amp * e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :]
    return rho


def _lognormal(c, seed):
    """exp of a Gaussian random field with a power-law spectrum, unit variance."""
    n, g = c["nx"], c["order"] // 2
    gen = torch.Generator(device=DEV)
    gen.manual_seed(int(seed))
    k = torch.fft.rfftn(torch.randn((n, n, n), dtype=torch.float64, device=DEV, generator=gen))
    fz = torch.fft.fftfreq(n, device=DEV, dtype=torch.float64) ** 2
    fx = torch.fft.rfftfreq(n, device=DEV, dtype=torch.float64) ** 2
    k2 = fz[:, None, None] + fz[None, :, None] + fx[None, None, :]
    k2[0, 0, 0] = 1.0
    k *= k2 ** (-11.0 / 12.0)
    del k2
    k[0, 0, 0] = 0.0
    f = torch.fft.irfftn(k, s=(n, n, n))
    del k
    f = torch.exp(f / f.std(unbiased=False) - 0.5)
    i = torch.arange(-(g - 1), n + g, device=DEV) % n
    return f[i][:, i][:, :, i].contiguous()


def _spheres(c, rng):
    """Two spheres of density (1 - w^2)^2."""
    x, y, z = _axes(c)
    rho = torch.zeros((z.numel(), y.numel(), x.numel()), dtype=torch.float64, device=DEV)
    for p in (0.35, 0.65):
        u, a = p + rng.uniform(-0.05, 0.05, 3), rng.uniform(0.1, 0.2)
        d2 = ((x - u[0]) ** 2)[None, None, :] + ((y - u[1]) ** 2)[None, :, None] + ((z - u[2]) ** 2)[:, None, None]
        rho += rng.uniform(0.5, 2.0) * torch.clamp(1.0 - d2 / a ** 2, min=0.0) ** 2
    return rho


def _ball(c, rng):
    """A uniform ball and its closed-form potential on the boundary nodes."""
    x, y, z = _axes(c)
    u, a = rng.uniform(0.45, 0.55, 3), rng.uniform(0.2, 0.3)
    r = torch.sqrt(((x - u[0]) ** 2)[None, None, :] + ((y - u[1]) ** 2)[None, :, None] + ((z - u[2]) ** 2)[:, None, None])
    phi = torch.where(r < a, 0.5 * PI4 * (r * r / 3.0 - a * a), -(PI4 / 3.0) * a ** 3 / torch.clamp(r, min=1e-300))
    _inside(phi, c["order"] // 2).zero_()
    return (r < a).to(torch.float64), phi


def _inside(t, g):
    return t[g:-g, g:-g, g:-g]


def _density(c, seed, shift=0.0):
    rng = np.random.default_rng(seed)
    if c["rho"] == "lognormal":
        return _lognormal(c, seed), None
    if c["rho"] == "spheres":
        return _spheres(c, rng), None
    if c["rho"] == "ball":
        return _ball(c, rng)
    return _blobs(c, rng, shift), None


def _solver(c):
    lo, hi = _box(c)
    return CartesianSolver((c["nx"], c["ny"], c["nz"]), order=c["order"], lo=lo, hi=hi, bc=c["bc"], lmax=c["lmax"])


def _solve(c, s, rho, phi):
    return s.solve(rho, phi, tol=c["tol"], method=c["method"], prec=c["prec"], omega=c["omega"], nu1=c["nu"],
                   nu2=c["nu"], max_iter=c["max_iter"], inner_cycles=c["inner"], sor_schedule=c["schedule"],
                   compact_order=c["compact"])


def _sph_grid(c):
    r = c["r_in"] * (1.0 / c["r_in"]) ** (np.arange(c["nr"]) / (c["nr"] - 1))
    th = (np.arange(c["nt"]) + 0.5) * math.pi / c["nt"]
    return r, th, 2.0 * math.pi * np.arange(c["np"]) / c["np"]


def _sph_density(c, seed):
    """r^-2 with a quadrupole in theta and an m = 2 bar in phi, of seeded strengths."""
    r, th, ph = _sph_grid(c)
    a, b, p0 = np.random.default_rng(seed).uniform([0.05, 0.1, 0.0], [0.15, 0.3, math.pi])
    rho = np.zeros((c["np"] + 2, c["nt"] + 2, c["nr"] + 2))
    rho[1:-1, 1:-1, 1:-1] = ((1.0 + a * np.cos(2.0 * (ph - p0)))[:, None, None]
                             * (1.0 + b * np.cos(th) ** 2)[None, :, None] * (r ** -2.0)[None, None, :])
    return torch.from_numpy(rho).to(DEV)


def _batch_member(c, n):
    return _cart("", (n, n, n), prec=c["prec"], inner=c["inner"], nu=c["nu"], tol=c["tol"], lmax=c["lmax"])


# ------------------------------------------------------------------ prepare and run
def prepare(case, seed):
    c = case
    if c["kind"] == "sph":
        r, th, ph = _sph_grid(c)
        rho = _sph_density(c, seed)
        return {"c": c, "s": SphericalSolver(r, th, ph, lmax=c["lmax"]), "rho": rho, "phi": torch.zeros_like(rho)}
    if c["kind"] == "batch":
        sizes = [int(v) for v in c["sizes"].split()]
        rhos = [_density(_batch_member(c, n), 1000 * (seed % 2 ** 31) + i)[0] for i, n in enumerate(sizes)]
        return {"c": c, "rhos": rhos, "phis": [torch.zeros_like(r) for r in rhos],
                "solvers": [CartesianSolver(n, bc="multipole", lmax=c["lmax"]) for n in sizes],
                "batch": Batch(len(sizes), max(sizes), prec=c["prec"], nu1=c["nu"], nu2=c["nu"],
                               inner_cycles=c["inner"])}
    rho, phi0 = _density(c, seed)
    st = {"c": c, "s": _solver(c), "rho": rho, "phi0": phi0, "phi": torch.zeros_like(rho)}
    if c["start"] == "warm":   # the potential of the previous step of a moving density
        prev, _ = _density(c, seed, shift=0.01)
        st["phi0"] = torch.zeros_like(rho)
        _solve(c, st["s"], prev, st["phi0"])
    return st


def run(state):
    c = state["c"]
    if c["kind"] == "sph":
        state["phi"].zero_()
        state["s"].solve(state["rho"], state["phi"], tol=c["tol"], prec=c["prec"], max_iter=c["max_iter"],
                         method=c["method"])
        return {"phi": state["phi"]}
    if c["kind"] == "batch":
        b, left = state["batch"], {}
        its = [0] * len(state["rhos"])
        for i, (s, rho, phi) in enumerate(zip(state["solvers"], state["rhos"], state["phis"])):
            phi.zero_()
            left[b.add(s, rho, phi, tol=c["tol"])] = i
        while left:
            b.step(c["step"])
            status, _ = b.poll()
            for slot in [q for q in left if status[q] != 0]:
                i = left.pop(slot)
                its[i] = b.remove(slot).iterations
        return {"phi": state["phis"], "iterations": its}
    if state["phi0"] is None:
        state["phi"].zero_()
    else:
        state["phi"].copy_(state["phi0"])
    info = _solve(c, state["s"], state["rho"], state["phi"])
    return {"phi": state["phi"], "iterations": info.iterations}


# ------------------------------------------------------------------ work
def _cart_work(c):
    """Density and starting potential read once, the potential written once (FP64);
    the arithmetic of the cycles the method needs to its tolerance: per cycle the
    smoothing sweeps, one residual and the transfers on all levels (8/7 of the
    finest)."""
    n = float((c["nx"] - 1) * (c["ny"] - 1) * (c["nz"] - 1))
    byt = 8.0 * (3.0 if c["start"] == "warm" or c["bc"] == "dirichlet" else 2.0) * n
    digits = -math.log10(c["tol"])
    taps = 27 if c["compact"] else (13 if c["order"] == 4 else 7)
    if c["method"] != "mg":
        steps = max(c["nx"], c["ny"], c["nz"]) * digits * (0.6 if c["method"] == "sor" else 0.3)
        return byt, steps * n * 3.0 * taps
    rate = {1: 0.9, 2: 1.15, 3: 1.5}[c["nu"]] if not c["compact"] else {1: 1.2, 2: 1.5, 3: 1.75}[c["nu"]]
    sweeps = 2 * c["nu"] * (2 if c["compact"] else 1) + 1
    return byt, math.ceil(digits / rate) * n * 8.0 / 7.0 * (sweeps * (taps + 1.0) + 6.0)


def work(case):
    c = case
    if c["kind"] == "sph":
        n = float(c["nr"] * c["nt"] * c["np"])
        return {"bytes": 16.0 * n, "flops": 400.0 * n * (2 * 15 + 20)}
    if c["kind"] == "batch":
        w = [_cart_work(_batch_member(c, int(v))) for v in c["sizes"].split()]
        return {"bytes": sum(v[0] for v in w), "flops": sum(v[1] for v in w)}
    byt, fl = _cart_work(c)
    return {"bytes": byt, "flops": fl}


# ------------------------------------------------------------------ the same results in plain 64-bit torch
def _harmonics(lmax, x, y, z):
    """(l, m, value) of the Schmidt semi-normalised real solid harmonics r^l S_lm."""
    r2 = x * x + y * y + z * z
    one = torch.ones_like(r2)
    cs = {0: (one, None)}   # sectoral (cos, sin) pairs
    c, s = one, torch.zeros_like(r2)
    for m in range(1, lmax + 1):
        f = 1.0 if m == 1 else math.sqrt((2.0 * m - 1.0) / (2.0 * m))
        c, s = f * (x * c - y * s), f * (x * s + y * c)
        cs[m] = (c, s)
    for m in range(lmax + 1):
        for part in cs[m]:
            if part is None:
                continue
            p0, p1 = None, part
            yield m, m, p1
            for l in range(m + 1, lmax + 1):
                t = (2.0 * l - 1.0) * z * p1
                if p0 is not None:
                    t = t - math.sqrt((l - 1.0) ** 2 - m * m) * r2 * p0
                p0, p1 = p1, t / math.sqrt(l * l - m * m)
                yield l, m, p1


def _open_boundary(c, rho, phi):
    """The multipole potential about the box centre on every node outside the unknowns."""
    g, lo_hi = c["order"] // 2, _box(c)
    x, y, z = (q - 0.5 * (lo_hi[0][a] + lo_hi[1][a]) for a, q in enumerate(_axes(c)))
    h3 = math.prod((lo_hi[1][a] - lo_hi[0][a]) / n for a, n in enumerate((c["nx"], c["ny"], c["nz"])))
    mom = None
    for k in range(g, z.numel() - g, 32):
        e = min(k + 32, z.numel() - g)
        w = rho[k:e, g:-g, g:-g] * h3
        X, Y, Z = x[None, None, g:-g], y[None, g:-g, None], z[k:e, None, None]
        q = torch.stack([(w * v).sum() for _, _, v in _harmonics(c["lmax"], X + 0 * w, Y + 0 * w, Z + 0 * w)])
        mom = q if mom is None else mom + q
    out = torch.ones(phi.shape, dtype=torch.bool, device=DEV)
    _inside(out, g).fill_(False)
    k, j, i = torch.nonzero(out, as_tuple=True)
    px, py, pz = x[i], y[j], z[k]
    r2 = px * px + py * py + pz * pz
    v = torch.zeros_like(r2)
    for q, (l, _, s) in zip(mom, _harmonics(c["lmax"], px, py, pz)):
        v -= q * s * r2 ** (-(2 * l + 1) / 2.0)
    phi[k, j, i] = v


def _shift(t, g, d):
    nz, ny, nx = t.shape
    return t[g + d[2]:nz - g + d[2], g + d[1]:ny - g + d[1], g + d[0]:nx - g + d[0]]


def _axis_modes(m, order):
    """Eigenvectors and eigenvalues of the one-axis second difference times h^2."""
    if order == 2:
        k = torch.arange(1, m + 1, dtype=torch.float64)
        v = math.sqrt(2.0 / (m + 1)) * torch.sin(math.pi / (m + 1) * k[:, None] * k[None, :])
        return v.to(DEV), (-4.0 * torch.sin(0.5 * math.pi * k / (m + 1)) ** 2).to(DEV)
    t = torch.diag(torch.full((m,), -2.5, dtype=torch.float64))
    t += torch.diag(torch.full((m - 1,), 4.0 / 3.0, dtype=torch.float64), 1)
    t += torch.diag(torch.full((m - 2,), -1.0 / 12.0, dtype=torch.float64), 2)
    w, v = torch.linalg.eigh(t.triu() + t.triu(1).T)
    return v.to(DEV), w.to(DEV)


def _exact_cart(c, seed):
    """The discrete solution itself, by diagonalising the operator axis by axis."""
    rho, phi0 = _density(c, seed)
    g = c["order"] // 2
    lo, hi = _box(c)
    n = (c["nx"], c["ny"], c["nz"])
    h = [(hi[a] - lo[a]) / n[a] for a in range(3)]
    phi = torch.zeros_like(rho) if phi0 is None else phi0
    if c["bc"] == "multipole":
        _open_boundary(c, rho, phi)
    modes = [_axis_modes(n[a] - 1, c["order"]) for a in range(3)]
    lam = [modes[0][1][None, None, :], modes[1][1][None, :, None], modes[2][1][:, None, None]]
    ax = ((1, 0, 0), (0, 1, 0), (0, 0, 1))
    neg = lambda d: tuple(-v for v in d)  # noqa: E731
    mul = lambda d, s: tuple(v * s for v in d)  # noqa: E731
    b = PI4 * _inside(rho, g)
    if c["compact"]:
        faces = [d for a in ax for d in (a, neg(a))]
        edges = [tuple(p[k] + q[k] for k in range(3)) for i in range(3) for j in range(i) for p in (ax[i], neg(ax[i]))
                 for q in (ax[j], neg(ax[j]))]
        corners = [(i, j, k) for i in (-1, 1) for j in (-1, 1) for k in (-1, 1)]
        w0, w1, w2, w3 = {2: (-6.0, 1.0, 0.0, 0.0), 4: (-4.0, 1 / 3.0, 1 / 6.0, 0.0),
                          6: (-128 / 30.0, 14 / 30.0, 3 / 30.0, 1 / 30.0)}[c["compact"]]
        f = PI4 * rho
        if c["compact"] == 4:
            b = 0.5 * b + sum(_shift(f, 1, d) for d in faces) / 12.0
        elif c["compact"] == 6:
            b = (67 / 120.0) * b + sum(_shift(f, 1, d) for d in faces) / 18.0 + sum(_shift(f, 1, d) for d in edges) / 90.0
            e = f   # one more layer on every side, continued by a cubic along its axis
            for a in (2, 1, 0):
                p = [e.narrow(a, i, 1) for i in range(4)] + [e.narrow(a, e.shape[a] - 1 - i, 1) for i in range(4)]
                e = torch.cat([4 * p[0] - 6 * p[1] + 4 * p[2] - p[3], e, 4 * p[4] - 6 * p[5] + 4 * p[6] - p[7]], a)
            b = b - sum(_shift(e, 2, mul(d, 2)) for d in faces) / 240.0
            del e
        del f
        ab = (w1 * sum(_shift(phi, 1, d) for d in faces) + w2 * sum(_shift(phi, 1, d) for d in edges)
              + w3 * sum(_shift(phi, 1, d) for d in corners)) / h[0] ** 2
        s = [v + 2.0 for v in lam]   # the sum of the two neighbours along an axis
        eig = (w0 + w1 * (s[0] + s[1] + s[2]) + w2 * (s[0] * s[1] + s[1] * s[2] + s[0] * s[2])
               + w3 * s[0] * s[1] * s[2]) / h[0] ** 2
    else:
        ab = 0.0
        for a in range(3):
            near = _shift(phi, g, ax[a]) + _shift(phi, g, neg(ax[a]))
            if g == 2:
                far = _shift(phi, g, mul(ax[a], 2)) + _shift(phi, g, mul(ax[a], -2))
                near = (16.0 * near - far) / 12.0
            ab = ab + near / h[a] ** 2
        eig = sum(lam[a] / h[a] ** 2 for a in range(3))
    u = b - ab   # the unknowns of phi are zero here, so ab holds the boundary data's share
    del ab, b
    vx, vy, vz = (m[0] for m in modes)
    u = torch.matmul(vy.T, torch.matmul(u, vx))
    u = torch.matmul(vz.T, u.reshape(u.shape[0], -1)).reshape(u.shape) / eig
    u = torch.matmul(vz, u.reshape(u.shape[0], -1)).reshape(u.shape)
    _inside(phi, g).copy_(torch.matmul(torch.matmul(vy, u), vx.T))
    return phi


def _exact_sph(c, seed):
    """Fourier modes in phi, then block elimination along r."""
    rn, thn, phn = _sph_grid(c)
    nr, nt, npp = c["nr"], c["nt"], c["np"]
    re = np.concatenate([[2 * rn[0] - rn[1]], rn, [rn[-1] ** 2 / rn[-2]]])
    dt, dp = math.pi / nt, 2.0 * math.pi / npp
    dr = 0.5 * (re[2:] - re[:-2])
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(DEV)  # noqa: E731
    rho = _sph_density(c, seed)[1:-1, 1:-1, 1:-1]
    r, th, ph = T(rn), T(thn), T(phn)
    P, TH = ph[:, None], th[None, :]
    ux, uy, uz = torch.sin(TH) * torch.cos(P), torch.sin(TH) * torch.sin(P), torch.cos(TH) + 0 * P
    w = rho * (r ** 2 * T(dr))[None, None, :] * torch.sin(TH)[:, :, None] * dt * dp
    ghost = torch.zeros((npp, nt), dtype=torch.float64, device=DEV)
    for l, _, s in _harmonics(c["lmax"], ux, uy, uz):
        ghost -= (w * s[:, :, None] * (r ** l)[None, None, :]).sum() * s / re[-1] ** (l + 1)
    up = (0.5 * (re[2:] + re[1:-1])) ** 2 / (re[2:] - re[1:-1]) / dr / rn ** 2
    dn = (0.5 * (re[1:-1] + re[:-2])) ** 2 / (re[1:-1] - re[:-2]) / dr / rn ** 2
    sf = np.sin(np.arange(nt + 1) * math.pi / nt)
    sf[0] = sf[-1] = 0.0
    st = np.sin(thn)
    ang = np.zeros((nt, nt))   # the theta part times r^2
    for j in range(nt):
        for q, f in ((j + 1, sf[j + 1]), (j - 1, sf[j])):
            if 0 <= q < nt:
                ang[j, q] += f / (st[j] * dt * dt)
                ang[j, j] -= f / (st[j] * dt * dt)
    f = torch.fft.rfft(PI4 * rho, dim=0)
    gk = torch.fft.rfft(ghost, dim=0)
    f[:, :, -1] -= up[-1] * gk
    mm = torch.arange(f.shape[0], dtype=torch.float64, device=DEV)
    azi = -(4.0 / dp ** 2) * torch.sin(0.5 * mm * dp) ** 2
    base = T(ang)[None] + torch.diag_embed(azi[:, None] / T(st)[None, :] ** 2)
    eye = torch.eye(nt, dtype=torch.float64, device=DEV)[None]
    rhs = torch.stack([f.real, f.imag], -1)   # (m, theta, r, 2)
    C, D = [], []
    for i in range(nr):
        a = base / rn[i] ** 2 - (up[i] + dn[i]) * eye
        u = up[i] + (dn[i] if i == 0 else 0.0)   # the mirror ghost at the inner edge
        d = rhs[:, :, i]
        if i > 0:
            a = a - dn[i] * C[-1]
            d = d - dn[i] * D[-1]
        inv = torch.linalg.inv(a)
        C.append(u * inv)
        D.append(inv @ d)
    x = [None] * nr
    x[-1] = D[-1]
    for i in range(nr - 2, -1, -1):
        x[i] = D[i] - C[i] @ x[i + 1]
    s = torch.stack(x, 2)
    out = torch.zeros((npp + 2, nt + 2, nr + 2), dtype=torch.float64, device=DEV)
    out[1:-1, 1:-1, 1:-1] = torch.fft.irfft(torch.complex(s[..., 0], s[..., 1]), n=npp, dim=0)
    out[1:-1, 1:-1, -1] = ghost
    return out


def exact(case, seed):
    c = case
    if c["kind"] == "sph":
        return {"phi": _exact_sph(c, seed)}
    if c["kind"] == "batch":
        sizes = [int(v) for v in c["sizes"].split()]
        return {"phi": [_exact_cart(_batch_member(c, n), 1000 * (seed % 2 ** 31) + i) for i, n in enumerate(sizes)],
                "iterations": [None] * len(sizes)}
    return {"phi": _exact_cart(c, seed), "iterations": None}
