"""Fields at the edge of what the fixed-point colour passes allow for.

Growth: guesses that alternate from node to node and right-hand sides as large as
the largest value, of the signs that make both grow from sweep to sweep, with the
most sweeps that the passes take, one and two V-cycles against the FP64 oracle
within the repository's bar for two FP64 evaluations, 1e-10 of the largest value
(an overflow would be off by the value itself).

Peak: a potential whose peak stands 10^3 to 10^4 above the rest, one V-cycle with
the fixed-point passes and one with the same passes in FP64 (a NaN on an unread box
corner selects them), each against the oracle, over all nodes and over the faint
ones alone: the fixed-point passes may not be further off than FP64's by more
than a factor of two, the scatter between two evaluations of equal precision."""
import numpy as np
import pytest

from oracle import solve as OS
from oracle.grid import cart_grid

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

N = (96, 112, 80)
HI = tuple(v / 64 for v in N)


def _ref(order, guess, rho, cycles, nu, hi):
    ref = guess.copy()
    OS.solve_cartesian(rho, ref, cart_grid(N, order, hi=hi), "mg", 0.0, max_iter=cycles, nu1=nu, nu2=nu)
    return ref


def _gpu(order, guess, rho, cycles, nu, hi):
    import paper_2605_03563_gb300 as P
    phi = torch.from_numpy(guess).to("cuda:0")
    with P.CartesianSolver(N, order, hi=hi) as s:
        info = s.solve(torch.from_numpy(rho).to("cuda:0"), phi, tol=0.0, max_iter=cycles, nu1=nu, nu2=nu)
    assert info.status in (P.capi.PS_NOT_CONVERGED, P.capi.PS_DIVERGED)
    return phi.cpu().numpy()


@pytest.mark.parametrize("order,nu,box", [(2, 3, "equal"), (2, 3, "unequal"), (2, 1, "equal"), (4, 2, "equal")])
@pytest.mark.parametrize("g", ["checker", "constant", "rows"])
@pytest.mark.parametrize("f", ["checker", "-checker", "constant", "-constant"])
def test_growth(order, nu, box, g, f):
    hi = HI if box == "equal" else (HI[0], 1.3 * HI[1], 0.8 * HI[2])
    gw = order // 2
    shape = tuple(v + 2 * gw - 1 for v in N[::-1])
    k, j, i = np.meshgrid(*(np.arange(s) for s in shape), indexing="ij")
    pattern = {"checker": 1.0 - 2.0 * ((i + j + k) % 2), "constant": np.ones(shape), "rows": 1.0 - 2.0 * (j % 2)}
    guess = pattern[g] * 1.9990234375
    d = sum((2.0 if order == 2 else 2.5) * (N[a] / hi[a]) ** 2 for a in range(3))
    rho = pattern[f.strip("-")] * (-1.0 if f[0] == "-" else 1.0) * 1.9990234375 * d / (4 * np.pi)
    for cycles in (1, 2):
        got, ref = _gpu(order, guess, rho, cycles, nu, hi), _ref(order, guess, rho, cycles, nu, hi)
        assert np.max(np.abs(got - ref)) <= 1e-10 * max(np.max(np.abs(ref)), np.max(np.abs(guess)))


@pytest.mark.parametrize("width", [0.002, 0.02])
@pytest.mark.parametrize("order,box", [(2, "equal"), (2, "unequal"), (4, "equal")])
def test_peak(order, box, width):
    hi = HI if box == "equal" else (HI[0], 1.3 * HI[1], 0.8 * HI[2])
    gw = order // 2
    shape = tuple(v + 2 * gw - 1 for v in N[::-1])
    z, y, x = np.meshgrid(*(np.linspace(0, 1, s) for s in shape), indexing="ij")
    r2 = (x - .4) ** 2 + (y - .5) ** 2 + (z - .6) ** 2
    guess = 1e4 * np.exp(-r2 / width) + 1.0 + 0.3 * np.sin(5 * x + 3 * y) * np.cos(4 * z)
    ref = _ref(order, guess, np.zeros(shape), 1, 1, hi)
    err = []
    for corner in (guess[0, 0, 0], np.nan):
        a = guess.copy()
        a[0, 0, 0] = corner
        e = np.abs(_gpu(order, a, np.zeros(shape), 1, 1, hi) - ref)
        e[0, 0, 0] = 0.0
        err.append([np.max(e), np.sqrt(np.mean(e ** 2)), np.sqrt(np.mean(e[guess < 10.0] ** 2))])
    for fixed, fp64 in zip(*err):
        assert fixed <= 2.0 * fp64, err
