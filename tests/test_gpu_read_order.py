"""State reads into memory that the device reaches come after the work already
queued there on the default stream, with a context on a stream that does not
wait for that one by itself: a fill of the output queued before the read does
not overwrite it, and a pinned buffer still being copied from keeps its old
rows for that copy.  A long kernel holds the default stream meanwhile."""
import ctypes as C

import numpy as np
import pytest

import fsi_cases as fc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import Simulation, lib  # noqa: E402

CASES = {
    "small": lambda: fc.tiny_box(seed=1),                            # all outputs in one copy
    "large": lambda: fc.tiny_box_3d(seed=1, n=(40, 32, 32)),         # one copy per output
}
BUSY = 200_000_000   # cycles, about 0.1 s


@pytest.mark.parametrize("call", ["fluid", "solid_positions"])
@pytest.mark.parametrize("kind", ["device", "pinned"])
@pytest.mark.parametrize("name", list(CASES))
def test_reads_follow_the_default_stream(name, kind, call):
    sim = Simulation.from_case(CASES[name](), stream=torch.cuda.Stream())
    sim.step()
    sim.sync()
    n = sim.nf if call == "fluid" else sim.ns
    want = (sim.get_fluid if call == "fluid" else sim.get_solid)()["r"]

    def read(buf):
        p = C.c_void_p(buf.data_ptr())
        rc = (lib().sphfsi_get_fluid(sim.h, p, None, None, None, None) if call == "fluid"
              else lib().sphfsi_get_solid_positions_all(sim.h, p))
        assert rc == 0

    if kind == "device":
        buf = torch.zeros((n, sim.dim), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        torch.cuda._sleep(BUSY)
        buf.fill_(-7.0)
        read(buf)
        torch.cuda.synchronize()
        assert np.array_equal(buf.cpu().numpy(), want)
    else:
        buf = torch.full((n, sim.dim), -7.0, dtype=torch.float64).pin_memory()
        copy = torch.zeros((n, sim.dim), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        torch.cuda._sleep(BUSY)
        copy.copy_(buf, non_blocking=True)
        read(buf)
        torch.cuda.synchronize()
        assert np.array_equal(buf.numpy(), want)
        assert bool((copy == -7.0).all())
    sim.close()
