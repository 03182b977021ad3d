"""A fluid particle whose position is not a number stops the context in the
step that meets it, in every form of the pair loops: its pairs must not drop
out of the sums unnoticed."""
import numpy as np
import pytest

import fsi_cases as fc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import SphError, Simulation  # noqa: E402

E_UNSTABLE = -5
FORMS = {"cells": {}, "compact": dict(compact=1), "cell_rows": dict(rows=1), "tiles": dict(tile=1),
         "rows": dict(list=1)}


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("dim", [2, 3])
def test_a_nan_position_is_an_unstable_step(dim, form):
    case = fc.tiny_box(seed=1) if dim == 2 else fc.tiny_box_3d(seed=1)
    case.n_reinit = 0
    sim = Simulation.from_case(case)
    sim.set_tuning(**{**dict(lanes=4, block=128, compact=0, tile=0, records=0, rows=0, list=0), **FORMS[form]})
    sim.step()
    sim.sync()
    for axis in range(dim):
        blob = sim.get_state()
        r = sim.get_fluid()["r"]
        r[sim.nf // 2, axis] = np.nan
        sim.set_fluid_state(r=r)
        sim.step()
        with pytest.raises(SphError) as e:
            sim.sync()
        assert e.value.code == E_UNSTABLE
        sim.set_state(blob)
        sim.step()
        sim.sync()
    sim.close()
