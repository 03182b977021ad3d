"""State reads beyond the staging buffer's 64 MB go out in ranges of rows: a
3-D tank of 1.3M fluid particles (78 MB of rows; two ranges) gives, in the
caller's order, the rows that reads of one output at a time (each within the
buffer) give, into host arrays and into device tensors; the device memory that reads
take is bounded by the buffer."""
import ctypes as C

import numpy as np
import pytest

import fsi_cases as fc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import Simulation, lib  # noqa: E402


@pytest.mark.parametrize("device", [False, True])
def test_rows_beyond_the_staging_buffer(device):
    case = fc.tiny_box_3d(seed=1, n=(130, 100, 100))
    sim = Simulation.from_case(case)
    n = sim.nf
    outs = [((n, 3), torch.float64), ((n, 3), torch.float32), ((n,), torch.float64), ((n,), torch.float32),
            ((n, 3), torch.float32)]
    row = [24, 12, 8, 4, 12]
    assert n * sum(row) > 64 << 20 > n * max(row)
    free = torch.cuda.mem_get_info()[0]
    assert np.array_equal(sim.get_fluid()["r"], case.f_r)
    assert free - torch.cuda.mem_get_info()[0] <= 66 << 20   # the buffer, in whole 2 MB pages
    sim.step()
    sim.sync()

    def read(asked):
        bufs = [torch.full(s, -7, dtype=t, device="cuda" if device else "cpu") if k in asked else None
                for k, (s, t) in enumerate(outs)]
        assert lib().sphfsi_get_fluid(sim.h, *[C.c_void_p(None if b is None else b.data_ptr()) for b in bufs]) == 0
        return [None if b is None else b.cpu().numpy() for b in bufs]

    whole = read(range(5))
    for k in range(5):
        assert np.array_equal(read([k])[k], whole[k]), k
    sim.close()
