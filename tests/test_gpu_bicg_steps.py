"""BiCGSTAB iterations in one cooperative launch against the kernels of an
iteration (a handle with kernel timing on runs those): potentials and iteration
counts bit for bit, on grids smaller and larger than a 32 x 8 x 8 tile, with
plane counts that are no multiple of a chunk, more warps of work than the
launch has, both inner boundaries and both precisions, and for a solve stopped
by max_iter and one advanced in several steps."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "mixed_fp32"])
@pytest.mark.parametrize("inner", ["neumann", "multipole"])
@pytest.mark.parametrize("nr,nt,npp", [(3, 2, 4), (12, 6, 8), (33, 9, 18), (64, 24, 12), (110, 48, 32), (130, 50, 32)])
def test_steps_equal_kernels(nr, nt, npp, inner, prec):
    import paper_2605_03563_gb300 as P
    r, th, ph = W.spherical_coords(nr, nt, npp, r_in=0.4 if nr == 3 else 0.1)
    rho = torch.from_numpy(W.spherical_density(r, th, ph)).to("cuda:0")
    with P.SphericalSolver(r, th, ph, lmax=2, inner=inner) as s:
        def run(max_iter, parts=None):
            phi = torch.zeros_like(rho)
            if parts is None:
                return s.solve(rho, phi, tol=1e-8, prec=prec, max_iter=max_iter), phi
            s.begin(rho, phi, tol=1e-8, method="bicgstab", prec=prec, max_iter=max_iter, inner_cycles=0)
            for k in parts:
                s.step(k)
            return s.end(), phi
        full, phi = run(400)
        cut, phc = run(7)
        stepped, phs = run(60, (1, 2, 19, 100))
        s.profile(True)
        ref, phr = run(400)
        refc, phrc = run(7)
        refs, phrs = run(60)
    assert (full.iterations, full.status, full.rel_residual) == (ref.iterations, ref.status, ref.rel_residual)
    assert (cut.iterations, cut.status) == (refc.iterations, refc.status)
    assert stepped.iterations == refs.iterations
    assert torch.equal(phi, phr) and torch.equal(phc, phrc) and torch.equal(phs, phrs)


@pytest.mark.parametrize("prec", ["fp64", "mixed_fp32"])
def test_handle_reused_with_another_density(prec):
    """A loop graph captured for one density buffer serves a solve of another."""
    import paper_2605_03563_gb300 as P
    r, th, ph = W.spherical_coords(160, 56, 40, r_in=0.1)   # above the one-launch size
    a = torch.from_numpy(W.spherical_density(r, th, ph)).to("cuda:0")
    b = torch.flip(a, (1,)).contiguous() * 3.0 + 1.0
    def solve(s, rho):
        phi = torch.zeros_like(rho)
        return s.solve(rho, phi, tol=1e-8, prec=prec, max_iter=3000), phi
    with P.SphericalSolver(r, th, ph, lmax=2) as s, P.SphericalSolver(r, th, ph, lmax=2) as fresh:
        solve(s, a)
        again, phi = solve(s, b)
        want, ref = solve(fresh, b)
    assert (again.iterations, again.status, again.rel_residual) == (want.iterations, want.status, want.rel_residual)
    assert torch.equal(phi, ref)
