"""The grid barrier of the one-launch iterations: every block sees all others'
writes behind it, also where the arrival counter passes 2^32; a barrier that
an arrival is missing from is given up after its limit by every block, sets the
fault flag and leaves the context usable."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("start", [0, 2 ** 32 - 1000, 2 ** 31 - 50])
@pytest.mark.parametrize("blocks", [1, 7, 0])
def test_blocks_stay_in_step(blocks, start):
    from paper_2605_03563_gb300 import capi, ops
    blocks = blocks or torch.cuda.get_device_properties(0).multi_processor_count
    out = torch.zeros(5 + blocks, dtype=torch.int32, device="cuda")
    st, _ = ops.probe_grid_barrier(blocks, 200, out, start=start)
    assert st == capi.PS_OK, capi.lib().poisson_last_error()
    got = out.cpu().numpy().view("uint32")
    assert int(got[0]) == (start + 200 * blocks) % 2 ** 32 and (got[5:] == 200).all()


def test_a_missing_arrival_is_reported_by_every_block():
    from paper_2605_03563_gb300 import capi, ops
    out = torch.zeros(12, dtype=torch.int32, device="cuda")
    st, ms = ops.probe_grid_barrier(7, 3, out, missing=True)
    assert st == capi.PS_ERR_TIMEOUT and 2000.0 <= ms < 4000.0, (st, ms)
    assert out[1] == 1 and out[3] == 7 and (out[5:] == 1).all()
    st, _ = ops.probe_grid_barrier(7, 3, out)
    assert st == capi.PS_OK
