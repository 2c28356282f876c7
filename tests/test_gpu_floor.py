"""How far a solve can converge from a source of one node, whose potential peaks
two hundred times above its r.m.s.: to the rounding of FP64 sums, not to the
units of the fixed-point passes.

The tolerance of each solve is derived from its own potential u: an FP64
residual rounds every term of A u once at the term's size, W |u| 2^-53 a node (W
the sum of the weights' magnitudes), so ||f - A u|| down to
2^-53 W ||u||_2 can be asked for.  Units of the largest value leave 2 to 5 times
that at these sizes."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,order,compact,prec", [
    ((192, 192, 192), 2, 0, "fp64"), ((192, 192, 192), 2, 0, "mixed_fp32"), ((192, 160, 176), 2, 0, "fp64"),
    ((192, 192, 192), 4, 0, "fp64"), ((160, 160, 160), 4, 0, "mixed_fp32"), ((192, 192, 192), 2, 6, "fp64"),
    ((192, 192, 192), 2, 6, "mixed_fp32"), ((192, 192, 192), 2, 2, "fp64")])
def test_point_source(n, order, compact, prec):
    import paper_2605_03563_gb300 as P
    g = order // 2
    shape = tuple(v + 2 * g - 1 for v in n[::-1])
    rho = torch.zeros(shape, dtype=torch.float64, device="cuda:0")
    rho[tuple(s // 2 for s in shape)] = 1.0
    h = [1.0 / v for v in n]
    w = 2 * {0: {2: 2.0, 4: 32 / 12}[order], 2: 2.0, 4: 4 / 3, 6: 128 / 90}[compact]   # per axis, in units of 1/h^2
    W = sum(w / v ** 2 for v in h)
    with P.CartesianSolver(n, order, bc="multipole", lmax=0) as s:
        def solve(tol):
            phi = torch.zeros(shape, dtype=torch.float64, device="cuda:0")
            info = s.solve(rho, phi, tol=tol, max_iter=40, prec=prec, nu1=2, nu2=2, compact_order=compact)
            return info, phi
        info, phi = solve(1e-8)
        assert info.converged
        ref = 4 * np.pi * {0: 1.0, 2: 1.0, 6: np.sqrt((67 / 120) ** 2 + 6 / 18 ** 2 + 12 / 90 ** 2 + 6 / 240 ** 2)}[compact]
        tol = 2.0 ** -53 * W * float(torch.linalg.norm(phi)) / ref
        info, phi = solve(tol)
    assert info.converged, (info.rel_residual, tol)
    assert 1e-16 < tol < 1e-14
