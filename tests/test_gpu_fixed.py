"""Residual passes whose neighbour sums run on the integer pipe: the relative
residual of a given guess (max_iter = 0), 7- and 13-point and compact 27-point,
against a plain FP64 evaluation, on a grid above the size from which these
passes are taken and ragged against their 64 x 16 tile, and just below that
size (the FP64 passes).  Guesses: smooth, random from node to node (second
differences as large as the values), one spike 1e8 above the rest, zero
inside non-zero boundary data, values near the lower end of the exponent
range (the march's FP64 form), and one infinity (divergence).

Tolerance, derived before the first run: a residual of r.m.s. r formed from
values of size U with the stencil's weights W (sum of magnitudes) may be off by
a few roundings of W U at every node, here 32 of them, 32 2^-53 W U / r
relative; the norms themselves add 1e-12.  The refinement's norm is summed in
FP32: 1e-5.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BIG, SMALL = (96, 112, 80), (80, 96, 64)


def _residual(u, f, h, order, compact):
    g = order // 2
    def sh(a, dx, dy, dz):
        nz, ny, nx = a.shape
        return a[g + dz:nz - g + dz, g + dy:ny - g + dy, g + dx:nx - g + dx]
    c = sh(u, 0, 0, 0)
    if compact:
        w = {2: (-6, 1, 0, 0), 4: (-4, 1 / 3, 1 / 6, 0), 6: (-128 / 30, 14 / 30, 3 / 30, 1 / 30)}[compact]
        acc = 0.0
        for dz in (-1, 0, 1):
            for dy in (-1, 0, 1):
                for dx in (-1, 0, 1):
                    acc = acc + w[abs(dx) + abs(dy) + abs(dz)] * sh(u, dx, dy, dz)
        return f - acc / h ** 2, sum(abs(w[k]) * n for k, n in enumerate((1, 6, 12, 8))) / h ** 2
    acc = 0.0
    for d in ((1, 0, 0), (0, 1, 0), (0, 0, 1)):
        n1 = sh(u, *d) + sh(u, *(-v for v in d))
        if order == 4:
            n2 = sh(u, *(2 * v for v in d)) + sh(u, *(-2 * v for v in d))
            acc = acc + (16 * n1 - n2 - 30 * c) / 12.0
        else:
            acc = acc + (n1 - 2 * c)
    return f - acc / h ** 2, (16.0 if order == 4 else 12.0) / h ** 2


def _guess(kind, shape, g):
    rng = np.random.Generator(np.random.PCG64(4))
    z, y, x = np.meshgrid(*(np.linspace(0, 1, s) for s in shape), indexing="ij")
    u = np.exp(-((x - .4) ** 2 + (y - .5) ** 2 + (z - .6) ** 2) / .1) - 2.0
    if kind == "rough":
        u = rng.standard_normal(shape)
    elif kind == "spike":
        u[shape[0] // 2, shape[1] // 3, shape[2] // 4] = 1e8
    elif kind == "boundary":
        u[g:-g, g:-g, g:-g] = 0.0
    elif kind == "tiny":
        u = u * 1e-270
    return u


@pytest.mark.parametrize("kind", ["smooth", "rough", "spike", "boundary", "tiny"])
@pytest.mark.parametrize("order,compact,prec", [(2, 0, "fp64"), (4, 0, "fp64"), (2, 0, "mixed_fp32"), (4, 0, "mixed_bf16"),
                                                (2, 2, "fp64"), (2, 4, "mixed_fp32"), (2, 6, "fp64"), (2, 6, "mixed_fp32")])
@pytest.mark.parametrize("n", [BIG, SMALL])
def test_initial_residual(n, order, compact, prec, kind):
    import paper_2605_03563_gb300 as P
    g, h = order // 2, 1.0 / 64
    hi = tuple(v * h for v in n)
    shape = tuple(n[a] + 2 * g - 1 for a in (2, 1, 0))
    u = _guess(kind, shape, g)
    u0 = u.copy()
    u0[g:-g, g:-g, g:-g] = 0.0
    f = np.zeros(tuple(s - 2 * g for s in shape))   # rho = 0: the residual is the operator's value
    r, W = _residual(u, f, h, order, compact)
    r0, _ = _residual(u0, f, h, order, compact)
    want = np.sqrt(np.sum((r / np.max(np.abs(r))) ** 2)) * np.max(np.abs(r)) / (
        np.sqrt(np.sum((r0 / np.max(np.abs(r0))) ** 2)) * np.max(np.abs(r0)))
    rms = np.sqrt(np.mean((r / np.max(np.abs(r))) ** 2)) * np.max(np.abs(r))
    tol = 32 * 2.0 ** -53 * W * np.max(np.abs(u)) / rms + (1e-12 if prec == "fp64" or compact else 1e-5)
    phi = torch.from_numpy(u).to("cuda:0")
    with P.CartesianSolver(n, order, hi=hi) as s:
        info = s.solve(torch.zeros_like(phi), phi, tol=0.0, max_iter=0, prec=prec, compact_order=compact)
    if kind == "tiny":   # the squares of the norm underflow in any FP64 evaluation
        assert info.status in (P.capi.PS_OK, P.capi.PS_NOT_CONVERGED, P.capi.PS_DIVERGED)
        return
    assert abs(info.rel_residual - want) <= tol * want, (info.rel_residual, want, tol)
    assert np.array_equal(phi.cpu().numpy(), u)


@pytest.mark.parametrize("order,compact", [(2, 0), (4, 0), (2, 6)])
def test_infinite_guess_diverges(order, compact):
    import paper_2605_03563_gb300 as P
    g, h = order // 2, 1.0 / 64
    shape = tuple(BIG[a] + 2 * g - 1 for a in (2, 1, 0))
    u = _guess("smooth", shape, g)
    u[40, 50, 60] = np.inf
    phi = torch.from_numpy(u).to("cuda:0")
    with P.CartesianSolver(BIG, order, hi=tuple(v * h for v in BIG)) as s:
        for prec in ("fp64", "mixed_fp32"):
            info = s.solve(torch.zeros_like(phi), phi, tol=1e-8, max_iter=3, prec=prec, compact_order=compact)
            assert info.status == P.capi.PS_DIVERGED


@pytest.mark.parametrize("compact", [2, 6])
def test_compact_fp64_solve_matches_oracle(compact):
    """A whole FP64 compact solve whose two finest levels take the fixed-point
    residual and SPAI passes (the second with Galerkin weights in integers):
    equal V-cycle counts, potentials within 1e-10 of the FP64 oracle."""
    import paper_2605_03563_gb300 as P
    import workloads as W
    from oracle import solve as OS
    from oracle.grid import cart_grid
    n, hi = (192, 176, 208), tuple(v / 192 for v in (192, 176, 208))
    x = [np.linspace(0, 1, v + 1) for v in n]
    rho = np.exp(-((x[0][None, None, :] - .4) ** 2 + (x[1][None, :, None] - .5) ** 2 + (x[2][:, None, None] - .6) ** 2) / .02)
    g = cart_grid(n, hi=hi)
    ref = g.zeros()
    info_o = OS.solve_cartesian(rho, ref, g, "mg", 1e-4, max_iter=10, bc="multipole", lmax=2, nu1=1, nu2=1,
                                compact_order=compact)
    phi = torch.zeros(W.cart_shape(n, 2), dtype=torch.float64, device="cuda:0")
    with P.CartesianSolver(n, hi=hi, bc="multipole", lmax=2) as s:
        info = s.solve(torch.from_numpy(rho).to("cuda:0"), phi, tol=1e-4, max_iter=10, nu1=1, nu2=1, compact_order=compact)
    assert info.iterations == info_o.iterations
    assert np.max(np.abs(phi.cpu().numpy() - ref)) <= 1e-10 * np.max(np.abs(ref))


@pytest.mark.parametrize("n,h,order,nu1,nu2", [
    ((96, 112, 80), (1, 1, 1), 2, 1, 1),          # 8-row tiles, lagged check
    ((176, 144, 144), (1, 1, 1), 2, 3, 2),        # 16-row tiles (above 3 10^6 nodes)
    ((176, 144, 144), (1, 1.25, 0.75), 2, 1, 2),  # unequal spacings, norm of colour 0
    ((112, 80, 96), (1, 0.75, 1.25), 2, 2, 3),
    ((192, 176, 208), (1, 1, 1), 2, 2, 1),        # the second level too
    ((96, 112, 80), (1, 1, 1), 4, 2, 2),          # 13-point
    ((144, 112, 112), (1, 1, 1), 4, 1, 2),
])
def test_fp64_solve_matches_oracle(n, h, order, nu1, nu2):
    """FP64 multigrid solves whose colour passes run on the integer pipe: equal
    V-cycle counts and potentials within 1e-10 of the FP64 oracle (the bound of
    solves that differ in rounding alone, as above), one V-cycle a step the
    same bits as the whole solve."""
    import paper_2605_03563_gb300 as P
    import workloads as W
    from oracle import solve as OS
    from oracle.grid import cart_grid
    hi = tuple(v * w / 128 for v, w in zip(n, h))
    g = order // 2
    x = [np.arange(1 - g, v + g) / v for v in n]
    rho = np.exp(-((x[0][None, None, :] - .4) ** 2 + (x[1][None, :, None] - .5) ** 2 + (x[2][:, None, None] - .6) ** 2) / .02)
    rho += 0.1 * np.random.Generator(np.random.PCG64(6)).standard_normal(rho.shape)
    ref = cart_grid(n, order, hi=hi).zeros()
    info_o = OS.solve_cartesian(rho, ref, cart_grid(n, order, hi=hi), "mg", 1e-4, max_iter=12, bc="multipole", lmax=2, nu1=nu1, nu2=nu2)
    rd = torch.from_numpy(rho).to("cuda:0")
    phi = torch.zeros(W.cart_shape(n, order), dtype=torch.float64, device="cuda:0")
    again = phi.clone()
    with P.CartesianSolver(n, order, hi=hi, bc="multipole", lmax=2) as s:
        info = s.solve(rd, phi, tol=1e-4, max_iter=12, nu1=nu1, nu2=nu2)
        s.begin(rd, again, tol=1e-4, max_iter=12, nu1=nu1, nu2=nu2)
        for _ in range(20):
            s.step(1)
        s.end()
    assert info.iterations == info_o.iterations
    assert torch.equal(phi, again)
    assert np.max(np.abs(phi.cpu().numpy() - ref)) <= 1e-10 * np.max(np.abs(ref))


@pytest.mark.parametrize("order", [4, 6])
@pytest.mark.parametrize("kind", ["smooth", "rough", "spike", "steps"])
@pytest.mark.parametrize("n", [(96, 112, 80), (160, 64, 96)])
def test_compact_right_hand_side(n, kind, order):
    """R_h on the integer pipe: the initial residual b - L_h phi of a solve from
    phi = 0 inside boundary data that make the reference norm known, against
    R_h rho evaluated in FP64 with the cubic extrapolation; the residual that
    is compared is ||b|| / ||b + boundary terms||, all of b.

    Tolerance, derived before the first run: b is formed from values truncated
    by less than 2^-56 of the largest (binade) with weights summing to 1.05, and
    the FP64 evaluation has 20 roundings: 32 2^-53 max|rho| / rms(b) relative."""
    import paper_2605_03563_gb300 as P
    h = 1.0 / 64
    shape = tuple(v + 1 for v in n[::-1])
    rho = _guess("smooth", shape, 1)
    rng = np.random.Generator(np.random.PCG64(9))
    if kind == "rough":
        rho = rng.standard_normal(shape)
    elif kind == "spike":
        rho[shape[0] // 2, shape[1] // 3, 0] = 1e7
    elif kind == "steps":
        rho = np.where(rng.random(shape) < 0.5, 1.0, -1e-3)
    f = np.pad(rho, 1)
    for ax in range(3):
        g = np.moveaxis(f, ax, 0)
        g[0] = 4 * g[1] - 6 * g[2] + 4 * g[3] - g[4]
        g[-1] = 4 * g[-2] - 6 * g[-3] + 4 * g[-4] - g[-5]
    def sh(dz, dy, dx):
        return f[2 + dz:f.shape[0] - 2 + dz, 2 + dy:f.shape[1] - 2 + dy, 2 + dx:f.shape[2] - 2 + dx]
    fa = ed = ax2 = 0.0
    for p in (-1, 1):
        fa = fa + sh(p, 0, 0) + sh(0, p, 0) + sh(0, 0, p)
        ax2 = ax2 + sh(2 * p, 0, 0) + sh(0, 2 * p, 0) + sh(0, 0, 2 * p)
        for q in (-1, 1):
            ed = ed + sh(p, q, 0) + sh(p, 0, q) + sh(0, p, q)
    b = sh(0, 0, 0) / 2 + fa / 12 if order == 4 else 67 / 120 * sh(0, 0, 0) + fa / 18 + ed / 90 - ax2 / 240
    b = 4 * np.pi * b
    # a guess v whose residual is compared: r = b - L_h v, the reference that of v's boundary alone (0 here: b)
    v = 1e-3 * _guess("smooth", shape, 1)
    v[0] = v[-1] = 0.0
    v[:, 0] = v[:, -1] = 0.0
    v[:, :, 0] = v[:, :, -1] = 0.0
    v *= np.max(np.abs(rho)) * h * h
    lv, W = _residual(v, np.zeros(tuple(s - 2 for s in shape)), h, 2, order)   # -L_h v
    want = np.linalg.norm(b + lv) / np.linalg.norm(b)
    tol = 32 * 2.0 ** -53 * (4 * np.pi * np.max(np.abs(rho)) + W * np.max(np.abs(v))) / np.sqrt(np.mean(b * b)) + 1e-12
    phi = torch.from_numpy(v).to("cuda:0")
    with P.CartesianSolver(n, hi=tuple(a * h for a in n)) as s:
        info = s.solve(torch.from_numpy(rho).to("cuda:0"), phi, tol=0.0, max_iter=0, compact_order=order)
    assert abs(info.rel_residual - want) <= tol * max(want, 1.0), (info.rel_residual, want, tol)
