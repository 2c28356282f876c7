"""R_h of the compact schemes node by node: bodies in vacuum, values of both signs
over 6 binades, a void 1e-12 of the body in it, a peak over a faint background,
Gaussian tails, subnormals, an infinity; on grids ragged against the kernels'
tiles.  Every node keeps the precision of its own neighbourhood.

Tolerance, derived before the first run: a node is a sum of at most 33 terms
(sixth order next to a corner: 27 with the extrapolations written out) formed with
fewer than 30 roundings, each of at most the sum of the terms' magnitudes L:
30 2^-53 L at that node, whatever the rest of the field holds; among subnormals
16 roundings of half the smallest one."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rhs(rho, order):
    """R_h rho and the sum of the terms' magnitudes, in extended precision."""
    r = rho.astype(np.longdouble)
    f, a = np.pad(r, 1), np.pad(np.abs(r), 1)
    for ax in range(3):
        for arr, sg in ((f, -1), (a, 1)):
            m = np.moveaxis(arr, ax, 0)
            m[0] = 4 * m[1] + sg * 6 * m[2] + 4 * m[3] + sg * m[4]
            m[-1] = 4 * m[-2] + sg * 6 * m[-3] + 4 * m[-4] + sg * m[-5]

    def sh(v, dz, dy, dx):
        return v[2 + dz:v.shape[0] - 2 + dz, 2 + dy:v.shape[1] - 2 + dy, 2 + dx:v.shape[2] - 2 + dx]
    out = []
    one = np.longdouble(1)
    for v, sg in ((f, -1), (a, 1)):
        fa = ed = ax2 = 0
        for p in (-1, 1):
            fa = fa + sh(v, p, 0, 0) + sh(v, 0, p, 0) + sh(v, 0, 0, p)
            ax2 = ax2 + sh(v, 2 * p, 0, 0) + sh(v, 0, 2 * p, 0) + sh(v, 0, 0, 2 * p)
            for q in (-1, 1):
                ed = ed + sh(v, p, q, 0) + sh(v, p, 0, q) + sh(v, 0, p, q)
        c = sh(v, 0, 0, 0)
        out.append(c / 2 + fa / 12 if order == 4 else one * 67 / 120 * c + fa / 18 + ed / 90 + sg * ax2 / 240)
    return out


def _density(kind, shape, rng):
    z, y, x = np.meshgrid(*(np.linspace(0, 1, s) for s in shape), indexing="ij")
    r2 = (x - .4) ** 2 + (y - .5) ** 2 + (z - .6) ** 2
    if kind == "bodies":
        return np.where(r2 < .04, 1.7, np.where((x - .8) ** 2 + (y - .8) ** 2 + (z - .3) ** 2 < .01, 0.3, 0.0))
    if kind == "signs":
        return rng.choice([-1.0, 1.0], shape) * rng.uniform(1 / 64, 2, shape) 
    if kind == "void":
        return np.where(r2 < .01, 1.0, 1e-12 * (1 + rng.random(shape)))
    if kind == "peak":
        rho = 1 + rng.random(shape)
        rho[shape[0] // 2, shape[1] // 3, 7] = 3.3e5
        return rho
    if kind == "gauss":
        return np.exp(-r2 / (2 * .03 ** 2))
    if kind == "subnormal":
        return np.where(r2 < .04, 1.0, 5e-324)
    if kind == "infinite":
        rho = 1 + rng.random(shape)
        rho[20, 30, 40] = np.inf
        return rho
    return np.zeros(shape)


@pytest.mark.parametrize("order", [4, 6])
@pytest.mark.parametrize("n,kind", [((96, 112, 80), k) for k in ("bodies", "signs", "void", "peak", "gauss",
                                                                 "subnormal", "infinite", "zero")] +
                         [((131, 70, 101), k) for k in ("signs", "peak")] + [((40, 36, 50), k) for k in ("signs", "void")])
def test_node_by_node(n, kind, order):
    import paper_2605_03563_gb300.ops as O
    rng = np.random.Generator(np.random.PCG64(17))
    rho = _density(kind, tuple(v + 1 for v in n[::-1]), rng)
    scale = 4 * np.pi
    b = torch.full(rho.shape, 7.0, dtype=torch.float64, device="cuda:0")
    O.compact_rhs(n, order, torch.from_numpy(rho).to("cuda:0"), b, scale=scale, hi=tuple(float(v) for v in n))
    got = b.cpu().numpy()
    with np.errstate(invalid="ignore"):
        want, mag = (scale * v for v in _rhs(rho, order))
        inner = got[1:-1, 1:-1, 1:-1]
        ok = np.isfinite(np.asarray(mag, dtype=np.float64))
        assert not np.isfinite(inner[~ok]).any()
        err = np.abs(inner[ok] - want[ok])
        tol = 30 * np.longdouble(2) ** -53 * mag[ok] + np.longdouble(2) ** -1071
        assert (err <= tol).all(), (float(np.max(err / np.maximum(tol, 1e-300))), int((err > tol).sum()))
    edge = np.ones(got.shape, bool)
    edge[1:-1, 1:-1, 1:-1] = False
    assert (got[edge] == 7.0).all()
