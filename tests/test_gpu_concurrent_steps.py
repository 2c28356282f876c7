"""Several solves in flight at once whose iterations run in one cooperative launch
each: handles on their own streams, advanced in turn and from several threads,
as many as fit beside each other and more (those steps take the loop graphs).
Potentials, iteration counts and residuals are those of each solve alone, bit
for bit; a solve that is alone again afterwards runs in one launch a step again."""
import threading

import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _make(kind, i):
    import paper_2605_03563_gb300 as P
    if kind == "sor":
        rho = torch.from_numpy(W.gaussian_blobs(56, seed=30 + i)).to("cuda:0")
        return P.CartesianSolver(56), rho, dict(method="sor", omega=1.8, tol=1e-7, max_iter=400)
    r, th, ph = W.spherical_coords(96, 48, 32)
    rho = torch.from_numpy(W.spherical_density(r, th, ph)).to("cuda:0") * (1.0 + 0.1 * i)
    return P.SphericalSolver(r, th, ph, lmax=4), rho, dict(method="bicgstab", tol=1e-7, max_iter=3000,
                                                           prec="fp64" if i % 2 == 0 else "mixed_fp32")


@pytest.mark.parametrize("kind", ["sor", "bicgstab"])
@pytest.mark.parametrize("count", [3, 9])
@pytest.mark.parametrize("threads", [False, True])
def test_together_as_alone(kind, count, threads):
    jobs = [_make(kind, i) for i in range(count)]

    def solve(i, phi):
        s, rho, kw = jobs[i]
        return s.solve(rho, phi, **kw)
    alone = [torch.zeros_like(j[1]) for j in jobs]
    want = [solve(i, alone[i]) for i in range(count)]
    phis = [torch.zeros_like(j[1]) for j in jobs]
    torch.cuda.synchronize()
    got = [None] * count
    if threads:
        def work(i):
            got[i] = solve(i, phis[i])
        pool = [threading.Thread(target=work, args=(i,)) for i in range(count)]
        for t in pool:
            t.start()
        for t in pool:
            t.join()
    else:
        for (s, rho, kw), phi in zip(jobs, phis):
            s.begin(rho, phi, **{**kw, "inner_cycles": 0} if kind == "bicgstab" else kw)
        live = list(range(count))
        while live:
            for i in live:
                jobs[i][0].step(50)
            live = [i for i in live if not jobs[i][0].poll()[0]]
        got = [s.end() for s, _, _ in jobs]
        # 9 launches of a quarter of the device each do not fit: loop graphs, of many kernels an iteration
        if count == 9:
            assert all(g.kernel_launches > 2 * w.iterations for g, w in zip(got, want))
    again = torch.zeros_like(jobs[0][1])
    last = solve(0, again)
    for i in range(count):
        assert (got[i].iterations, got[i].status, got[i].rel_residual) == (want[i].iterations, want[i].status, want[i].rel_residual)
        assert torch.equal(phis[i], alone[i])
    assert torch.equal(again, alone[0]) and last.kernel_launches == want[0].kernel_launches < want[0].iterations
    for s, _, _ in jobs:
        s.close()
