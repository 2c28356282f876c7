"""Box edges and corners that an operator does not read may hold anything: a
solve whose guess carries a large sentinel (or NaN) there gives the bits (for
NaN: the values) of one that carries zeros, over the fixed-point passes of FP64
multigrid, refinement and the compact schemes.  The 7- and 13-point operators
and the compact scheme of second order read the face layers alone, of fourth
order the edges too."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = (96, 112, 80)
HI = tuple(v / 64 for v in N)


def _outside(shape, g):
    """Number of coordinates outside the interior, per node."""
    out = np.zeros(shape, int)
    for ax, s in enumerate(shape):
        i = np.arange(s)
        o = ((i < g) | (i >= s - g)).astype(int)
        out += o.reshape([-1 if a == ax else 1 for a in range(3)])
    return out


@pytest.mark.parametrize("order,compact,prec,nu1,nu2", [
    (2, 0, "fp64", 2, 2), (2, 0, "fp64", 0, 2), (4, 0, "fp64", 2, 2), (2, 0, "mixed_fp32", 2, 2),
    (4, 0, "mixed_bf16", 2, 2), (2, 2, "fp64", 2, 1), (2, 4, "fp64", 1, 2), (2, 4, "mixed_fp32", 2, 2)])
@pytest.mark.parametrize("box", ["equal", "unequal"])
def test_guess(order, compact, prec, nu1, nu2, box):
    import paper_2605_03563_gb300 as P
    if compact and box == "unequal":
        return   # compact schemes take equal spacings
    hi = HI if box == "equal" else (HI[0], 1.3 * HI[1], 0.8 * HI[2])
    g = order // 2
    shape = tuple(n + 2 * g - 1 for n in N[::-1])
    rng = np.random.Generator(np.random.PCG64(3))
    z, y, x = np.meshgrid(*(np.linspace(0, 1, s) for s in shape), indexing="ij")
    rho = np.exp(-((x - .4) ** 2 + (y - .5) ** 2 + (z - .6) ** 2) / .02) + 0.1 * rng.standard_normal(shape)
    guess = np.cos(3 * x + y) - z
    unread = _outside(shape, g) > max(compact // 2, 1)
    guess[unread] = 0.0

    def solve(a):
        phi = torch.from_numpy(a).to("cuda:0")
        with P.CartesianSolver(N, order, hi=hi) as s:
            info = s.solve(torch.from_numpy(rho).to("cuda:0"), phi, tol=1e-9, max_iter=40, prec=prec, nu1=nu1, nu2=nu2,
                           compact_order=compact)
        out = phi.cpu().numpy()
        assert np.array_equal(out[unread], a[unread], equal_nan=True)
        return info, np.where(unread, 0.0, out)
    ref, want = solve(guess)
    assert ref.converged
    a = guess.copy()
    a[unread] = 1e30 * np.where(rng.random(int(unread.sum())) < 0.5, 1.0, -1.0)
    info, got = solve(a)
    assert info.iterations == ref.iterations and np.array_equal(got, want)
    if not compact:   # (a 27-point pass multiplies by zero weights, which keeps a NaN)
        a[unread] = np.nan
        info, got = solve(a)
        assert info.iterations == ref.iterations
        assert np.max(np.abs(got - want)) <= (1e-10 if prec == "fp64" else 1e-8) * np.max(np.abs(want))


@pytest.mark.parametrize("order,prec", [(4, "fp64"), (6, "fp64"), (6, "mixed_fp32")])
def test_density(order, prec):
    """The same for the density of a compact solve: R_h of fourth order reads the
    centre and the faces, of sixth order the edges and the nodes at distance 2."""
    import paper_2605_03563_gb300 as P
    shape = tuple(n + 1 for n in N[::-1])
    rng = np.random.Generator(np.random.PCG64(5))
    rho = np.where(rng.random(shape) < 0.3, 1.0, 0.25)   # (exact in fixed point as well)
    unread = _outside(shape, 1) > (1 if order == 4 else 2)
    rho[unread] = 0.0

    def solve(a):
        phi = torch.zeros(shape, dtype=torch.float64, device="cuda:0")
        with P.CartesianSolver(N, hi=HI) as s:
            info = s.solve(torch.from_numpy(a).to("cuda:0"), phi, tol=1e-8, max_iter=30, prec=prec, compact_order=order)
        return info, phi.cpu().numpy()
    ref, want = solve(rho)
    assert ref.converged
    a = rho.copy()
    a[unread] = -1e30
    info, got = solve(a)
    assert info.iterations == ref.iterations and np.array_equal(got, want)
