"""A wait of the windowed sub-step kernel that gives up (its limit set to one
poll: 32 CTAs here, 24 sub-steps of two exchanges each) while more steps are
queued behind it, one by one or as graph replays: the step that timed out is
the last that ran, the sync reports it, and a restored checkpoint steps on bit
for bit like a context that never timed out."""
import numpy as np
import pytest

import fsi_cases as fc
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import SphError, Simulation  # noqa: E402

E_TIMEOUT = -6


@pytest.mark.parametrize("queue", ["steps", "graph"])
def test_steps_queued_behind_a_time_out_do_nothing(queue):
    case = fc.cantilever(L=124 * 0.005, t=8 * 0.005, dpS=0.005)   # 1024 particles, no fluid
    _, _, dts = O.OracleSim(case).suggest_dt()
    K, dt = 24, 23.5 * dts

    def make():
        sim = Simulation.from_case(case, stream=torch.cuda.Stream())
        sim.set_solid_path(2)
        sim.set_substeps(K)
        return sim

    sim, other = make(), make()
    for s in (sim, other):
        s.step(dt)
        s.sync()
    assert sim.info()["solid_path"] == 2
    blob = sim.get_state()
    sim.set_wait_limit(1)
    if queue == "steps":
        for _ in range(4):
            sim.step(dt)
    else:
        sim.run(4, dt)
    with pytest.raises(SphError) as e:
        sim.sync()
    assert e.value.code == E_TIMEOUT
    assert sim.info()["step"] == 2
    sim.set_wait_limit(0)
    sim.set_state(blob)
    for s in (sim, other):
        for _ in range(3):
            s.step(dt)
        s.sync()
    a, b = sim.get_solid(), other.get_solid()
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    sim.close()
    other.close()
