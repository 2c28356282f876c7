"""Coarsest-level CG on slabs of a thread-block cluster: grids whose coarsest
level has one plane per CTA, several, fewer planes than CTAs, its longest axis
along x, y or z, and more in-plane unknowns than threads; 7- and 13-point, equal
and unequal spacings, solo and batched, against the FP64 oracle (the
repository's bars: equal V-cycle counts, potentials within 1e-10; a batch
against the solo solve within 1e-12)."""
import numpy as np
import pytest

import workloads as W
from oracle import solve as OS
from oracle.grid import cart_grid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

GRIDS = [((16, 16, 16), 2, "equal"), ((32, 32, 32), 4, "equal"), ((18, 18, 34), 2, "equal"),
         ((24, 16, 208), 2, "equal"), ((208, 16, 24), 2, "equal"), ((16, 208, 16), 4, "equal"),
         ((40, 28, 52), 2, "unit"), ((42, 42, 42), 2, "equal"), ((36, 34, 38), 4, "unit")]


@pytest.mark.parametrize("n,order,box", GRIDS)
def test_coarse_cg_shapes(n, order, box):
    import paper_2605_03563_gb300 as P
    hi = (1.0, 1.0, 1.0) if box == "unit" else tuple(v / 16.0 for v in n)
    rho = W.rng(7).uniform(0.5, 1.5, W.cart_shape(n, order))
    g = cart_grid(n, order=order, hi=hi)
    ref = g.zeros()
    # a few cycles: what the coarsest level returns enters every one of them
    info_o = OS.solve_cartesian(rho, ref, g, "mg", 1e-6, max_iter=12, bc="multipole", lmax=2)
    rho_t = torch.from_numpy(rho).to("cuda:0")
    phi = torch.zeros_like(rho_t)
    phb = torch.zeros_like(rho_t)
    with P.CartesianSolver(n, order, hi=hi, bc="multipole", lmax=2) as s:
        info = s.solve(rho_t, phi, tol=1e-6, max_iter=12)
        with P.Batch(2, max(n), order=order) as b:
            slot = None
            if np.prod([v // 2 ** _halvings(n) - 1 for v in n]) <= 4096:   # what a batch accepts
                slot = b.add(s, rho_t, phb, tol=1e-6, max_iter=12)
                b.step(12)
                b.poll()
                ib = b.remove(slot)
    assert info.iterations == info_o.iterations
    scale = np.max(np.abs(ref))
    assert np.max(np.abs(phi.cpu().numpy() - ref)) <= 1e-10 * scale
    if slot is not None:
        assert ib.iterations == info.iterations
        assert np.max(np.abs((phb - phi).cpu().numpy())) <= 1e-12 * scale


def _halvings(n):
    k = 0
    while all(v % 2 == 0 and v >= 16 for v in n):
        n = tuple(v // 2 for v in n)
        k += 1
    return k
