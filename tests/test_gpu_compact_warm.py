"""FP64 compact solves started from a guess whose interior is far above its
boundary data, on a grid whose finest level takes the fixed-point passes: the
first residual of the first V-cycle needs the guess's own bound, not the
boundary's.  One V-cycle and a whole solve against the FP64 oracle.

Tolerance, derived before the first run: the two differ in rounding alone; a
V-cycle forms values of the size U of its input in fewer than 100 operations
that touch a node, each within a few roundings of U, 400 2^-53 U < 5e-14 U; a
whole solve is within the repository's bar of 1e-10."""
import numpy as np
import pytest

import workloads as W
from oracle import solve as OS
from oracle.grid import cart_grid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = (96, 112, 80)
HI = tuple(v / 64 for v in N)


@pytest.mark.parametrize("boundary", [0.0, 1e-3])
@pytest.mark.parametrize("order,nu1,nu2", [(2, 1, 1), (6, 2, 1), (4, 0, 2)])
def test_guess_above_its_boundary(order, nu1, nu2, boundary):
    import paper_2605_03563_gb300 as P
    x = [np.linspace(0, 1, v + 1) for v in N]
    bump = (np.sin(np.pi * x[0])[None, None, :] * np.sin(np.pi * x[1])[None, :, None] * np.sin(np.pi * x[2])[:, None, None])
    guess = boundary + 50.0 * bump + 0.1 * np.sin(9 * np.pi * x[0])[None, None, :] * bump
    edge = np.ones(guess.shape, bool)
    edge[1:-1, 1:-1, 1:-1] = False
    guess[edge] = boundary
    rho = np.exp(-((x[0][None, None, :] - .4) ** 2 + (x[1][None, :, None] - .5) ** 2 + (x[2][:, None, None] - .6) ** 2) / .02)
    grid = cart_grid(N, hi=HI)
    for max_iter, tol, bar in ((1, 0.0, 5e-14), (40, 1e-8, 1e-10)):
        ref = guess.copy()
        info_o = OS.solve_cartesian(rho, ref, grid, "mg", tol, max_iter=max_iter, nu1=nu1, nu2=nu2, compact_order=order)
        phi = torch.from_numpy(guess).to("cuda:0")
        with P.CartesianSolver(N, hi=HI) as s:
            info = s.solve(torch.from_numpy(rho).to("cuda:0"), phi, tol=tol, max_iter=max_iter, nu1=nu1, nu2=nu2,
                           compact_order=order)
        assert info.iterations == info_o.iterations
        assert np.max(np.abs(phi.cpu().numpy() - ref)) <= bar * np.max(np.abs(guess))
