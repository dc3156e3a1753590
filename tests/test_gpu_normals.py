"""The normals of the Philox stream: every remainder of a block of four and
outputs that are only 8-byte aligned give the same bits as a whole, aligned
call (the values themselves are checked against the oracle elsewhere)."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

import workloads  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count,shift", [(1, 0), (2, 0), (3, 1), (4, 1), (5, 0), (7, 1), (400003, 0), (100002, 1)])
def test_normals_of_any_count_and_alignment(count, shift):
    import paper_1901_06427_gb300.binding as B
    g = B.grid_for(workloads.small_case(n=(8, 8, 8), n_bodies=1))
    whole = g.philox_normals(1234567, 9, 2, 1, (count + 3) // 4 * 4)
    out = torch.full((count + 2,), float("nan"), dtype=torch.float64, device="cuda")
    st = B.lib().rbfib_philox_normals(g._h, 1234567, 9, 2, 1, count, ctypes.c_void_p(out.data_ptr() + 8 * shift))
    assert st == B.OK
    torch.cuda.synchronize()
    assert torch.equal(out[shift:shift + count], whole[:count])
    assert torch.isnan(out[:shift]).all() and torch.isnan(out[shift + count:]).all()
