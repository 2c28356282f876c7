"""FP32 and BF16 13-point colour passes over staged planes, through the sweep
operator on grids whose rows are 16-byte multiples (the staged passes) and not
(the per-node pass), above the size from which they are taken and ragged
against their 96 x 16 tile: one sweep against the three colour updates in FP64
arithmetic rounded once to the storage type.

Tolerance, derived before the first run: a value formed in FP32 from 14 terms of
size U is within 14 roundings, 14 2^-24 x 2 U (the weights' magnitudes sum to
below 2); later colours read values off by as much: x 3.  BF16 adds the storage
rounding of the value and of those it reads, 2^-8 U each way: x 3 as well.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["float32", "bfloat16"])
@pytest.mark.parametrize("n,hi", [((101, 107, 113), (1, 1, 1)), ((125, 90, 101), (1, 0.7, 0.9)), ((102, 107, 113), (1, 1, 1)),
                                  ((197, 98, 66), (2, 1, 0.66))])
def test_sweep(n, hi, dtype):
    import paper_2605_03563_gb300.ops as O
    rng = np.random.Generator(np.random.PCG64(11))
    shape = tuple(v + 3 for v in n[::-1])
    dt = getattr(torch, dtype)
    phi = torch.from_numpy(rng.standard_normal(shape)).to(dt)
    h = [hi[a] / n[a] for a in range(3)]
    f = torch.from_numpy(rng.standard_normal(shape) / min(h) ** 2).to(dt)
    dev_phi = phi.to("cuda:0")
    O.sweep(n, 4, dev_phi, f.to("cuda:0"), hi=hi)
    u, ff = phi.double().numpy(), f.double().numpy()
    diag = sum(30.0 / (12.0 * v * v) for v in h)
    k, j, i = np.meshgrid(*(np.arange(s) - 1 for s in shape), indexing="ij")
    col = (i + j + k) % 3
    I = (slice(2, -2),) * 3
    def sh(a, ax, s):
        ix = [slice(2, -2)] * 3
        ix[2 - ax] = slice(2 + s, a.shape[2 - ax] - 2 + s)
        return a[tuple(ix)]
    for c in range(3):
        v = sum((16 * (sh(u, a, 1) + sh(u, a, -1)) - (sh(u, a, 2) + sh(u, a, -2))) / (12 * h[a] ** 2) for a in range(3))
        gs = (v - ff[I]) / diag
        gs = torch.from_numpy(gs).to(dt).double().numpy()
        u[I] = np.where(col[I] == c, gs, u[I])
    got = dev_phi.double().cpu().numpy()
    U = np.max(np.abs(u))
    tol = 3 * (14 * 2.0 ** -23 + (2.0 ** -7 if dtype == "bfloat16" else 0.0)) * U
    assert np.max(np.abs(got - u)) <= tol
    edge = np.ones(shape, bool)
    edge[I] = False
    assert np.array_equal(got[edge], phi.double().numpy()[edge])
