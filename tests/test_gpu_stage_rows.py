"""Stage times of a step whose neighbour rows are built behind the start of the
solid branch (a dam break with a body beyond one cluster): the rows are stage 7
and no part of momentum."""
import pytest

import fsi_cases as fc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import Simulation  # noqa: E402


def test_rows_behind_the_fork_are_their_own_stage():
    sim = Simulation.from_case(fc.dam_gate(seed=1, dpF=5e-4), stream=torch.cuda.Stream())   # 56k particles, body of 6400
    assert sim.tuning()["list"] == 1
    sim.run(3)
    sim.sync()
    sim.set_profiling(True)
    rows = []
    for _ in range(5):
        sim.run(1)
        sim.sync()
        rows.append(sim.stage_times()["neighbour_rows"])
    # the build takes 12 us on 10k particles; two events back to back are 2 us apart
    assert sorted(rows)[2] > 5e-3, rows
    sim.close()
