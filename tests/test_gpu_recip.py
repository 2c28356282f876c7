"""The reciprocal behind the coarsest CG's scalars against 1 / x: within one unit
in the last place over the range that the CG lets through (|x| from 1e-280 to
1e280), at both signs, at powers of two (exact) and just beside them.

Derived: PTX bounds the approximation's relative error by 2^-20 at worst; two
Newton steps leave 2^-80 of it and the rounding of the last fused step, half a
unit, plus that of the residual 1 - x y, below 2^-52 of itself."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_within_one_unit():
    import paper_2605_03563_gb300.ops as O
    rng = np.random.Generator(np.random.PCG64(21))
    x = np.exp(rng.uniform(np.log(1e-280), np.log(1e280), 400000)) * rng.choice([-1.0, 1.0], 400000)
    m = rng.uniform(1, 2, 400000)
    p = 2.0 ** np.arange(-930, 931)
    x = np.concatenate([x, m, p, -p, np.nextafter(p, 0), np.nextafter(p, np.inf), [3.0, 1 / 3, 0.1, 10.0]])
    y = torch.empty(x.size, dtype=torch.float64, device="cuda:0")
    O.probe_recip(torch.from_numpy(x).to("cuda:0"), y)
    got, want = y.cpu().numpy(), 1.0 / x
    assert np.max(np.abs(got - want) / np.spacing(np.abs(want))) <= 1.0
    assert np.array_equal(got[800000:800000 + 2 * p.size], want[800000:800000 + 2 * p.size])
