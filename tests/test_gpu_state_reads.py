"""State reads through the C-ABI: every output alone equals the same output of
a read of all (bit for bit), into host arrays and into device tensors, below
and above the size up to which a read's outputs travel in one copy, and for an
instance of a batch; the rows are the caller's order (fluid at its initial
positions)."""
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
    "small_2d": lambda: [fc.tiny_box(seed=1)],
    "one_megabyte_2d": lambda: [fc.dam_gate(seed=1, dpF=6e-4)],        # 38k particles: 1.7 MB of fluid rows
    "small_3d": lambda: [fc.tiny_box_3d(seed=1)],
    "large_3d": lambda: [fc.tiny_box_3d(seed=1, n=(40, 32, 32))],      # a solid read above 1 MB, fluid 2.7 MB
    "batch": lambda: [fc.tiny_box(seed=2), fc.channel_flag(seed=1), fc.tiny_box(seed=3, nx=10, ny=14)],
}


def _outputs(sim):
    d, nf, ns = sim.dim, sim.nf, sim.ns
    fluid = [((nf, d), np.float64), ((nf, d), np.float32), ((nf,), np.float64), ((nf,), np.float32),
             ((nf, d), np.float32)]
    solid = [((ns, d), np.float64), ((ns, d), np.float32), ((ns, d, d), np.float64), ((ns, d), np.float64),
             ((ns, d), np.float64), ((ns, d), np.float32), ((ns, d), np.float32)]
    return ("sphfsi_get_fluid", fluid), ("sphfsi_get_solid", solid)


@pytest.mark.parametrize("name", list(CASES))
def test_every_output_alone_and_on_the_device(name):
    cases = CASES[name]()
    sim = Simulation.from_cases(cases)
    for b, case in enumerate(cases):
        sim.select(b)
        assert np.array_equal(sim.get_fluid()["r"], case.f_r)
        assert np.array_equal(sim.get_solid()["r"], case.s_r0)
    for _ in range(2):
        sim.step()
    sim.sync()
    for b in range(len(cases)):
        sim.select(b)
        for (fn, outs), whole in zip(_outputs(sim), (sim.get_fluid(), sim.get_solid())):
            want = list(whole.values())
            assert [w.shape for w in want] == [s for s, _ in outs]
            for device in (False, True):
                for k in list(range(len(outs))) + [None]:
                    bufs = [torch.from_numpy(np.full(s, -7, t)) if k is None or j == k else None
                            for j, (s, t) in enumerate(outs)]
                    if device:
                        bufs = [x if x is None else x.cuda() for x in bufs]
                        torch.cuda.synchronize()
                    ptr = [C.c_void_p(None if x is None else x.data_ptr()) for x in bufs]
                    assert getattr(lib(), fn)(sim.h, *ptr) == 0
                    for x, w in zip(bufs, want):
                        assert x is None or np.array_equal(x.cpu().numpy(), w), (name, fn, k, device)
    sim.close()
