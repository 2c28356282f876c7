"""The reference norm ||b - A u0|| of compact solves where it is far below ||b||: a
density on the first and last layers alone that the boundary data cancel but for
one part in 10^9.  From a zero guess the relative residual is 1.

Tolerance, derived before the first run: the norm and the residual's norm are sums of
the same numbers, each from b and A u0 of size b with a few roundings, 8 2^-53 b
against 10^-9 b: 1e-6."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed_fp32"])
@pytest.mark.parametrize("n", [(96, 112, 80), (64, 48, 32)])
def test_cancelling_layers(n, prec):
    import paper_2605_03563_gb300 as P
    shape = tuple(v + 1 for v in n[::-1])
    phi = np.zeros(shape)
    for ax in range(3):
        f = np.moveaxis(phi, ax, 0)
        f[0] = f[-1] = 1.0
    nb = np.zeros(shape)   # boundary neighbours of a node, second order's cross
    for ax, s in enumerate(shape):
        i = np.arange(s)
        nb = nb + ((i == 1) | (i == s - 2)).astype(float).reshape([-1 if a == ax else 1 for a in range(3)])
    edge = np.ones(shape, bool)
    edge[1:-1, 1:-1, 1:-1] = False
    rho = np.where(edge, 0.0, nb * (1.0 + 1e-9) / (4 * np.pi))   # spacing 1: A u0 = nb
    p = torch.from_numpy(phi).to("cuda:0")
    with P.CartesianSolver(n, hi=tuple(float(v) for v in n)) as s:
        info = s.solve(torch.from_numpy(rho).to("cuda:0"), p, tol=0.0, max_iter=0, prec=prec, compact_order=2)
    assert abs(info.rel_residual - 1.0) <= 1e-6, info.rel_residual
