"""SOR steps in one cooperative launch against the colour passes (a handle with
kernel timing on runs those): potentials bit for bit, equal step counts, over
the sizes at which the launch changes (block widths, more pairs than threads,
odd and even rows, one interior node), equal and unequal spacings, every weight
schedule, a solve stopped by max_iter and one advanced in several steps."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(2, 2, 2), (3, 4, 2), (33, 20, 18), (42, 43, 44), (45, 44, 43), (56, 54, 52), (101, 98, 97), (112, 96, 104)]


@pytest.mark.parametrize("box", ["equal", "unit"])
@pytest.mark.parametrize("schedule,omega", [("fixed", 1.0), ("fixed", 1.7), ("chebyshev", 1.0), ("optimal", 1.0)])
@pytest.mark.parametrize("n", SIZES)
def test_steps_equal_colour_passes(n, schedule, omega, box):
    import paper_2605_03563_gb300 as P
    hi = (1.0, 1.0, 1.0) if box == "unit" else tuple(v / 64.0 for v in n)
    g = W.rng(11)
    rho = torch.from_numpy(g.uniform(-1, 1, W.cart_shape(n, 2))).to("cuda:0")
    guess = torch.from_numpy(g.uniform(-1, 1, W.cart_shape(n, 2))).to("cuda:0")
    kw = dict(tol=1e-6, method="sor", omega=omega, sor_schedule=schedule)
    with P.CartesianSolver(n, hi=hi) as s:
        def run(max_iter):
            phi = guess.clone()
            return s.solve(rho, phi, max_iter=max_iter, **kw), phi
        one, phi = run(37)
        cut, phc = run(5)
        parts = guess.clone()
        s.begin(rho, parts, max_iter=37, **kw)
        for k in (1, 3, 40):
            s.step(k)
        stepped = s.end()
        s.profile(True)
        ref, phr = run(37)
        refc, phrc = run(5)
    assert (one.iterations, one.status) == (ref.iterations, ref.status)
    assert (cut.iterations, cut.status) == (refc.iterations, refc.status)
    assert torch.equal(phi, phr) and torch.equal(phc, phrc)
    assert stepped.iterations == ref.iterations and torch.equal(parts, phr)
    assert abs(one.rel_residual - ref.rel_residual) <= 1e-12 * ref.rel_residual
