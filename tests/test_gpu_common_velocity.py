"""A body and the fluid around it moving together at one velocity, without
pressure, gravity or walls: no pair has a relative velocity, so the density
rates and forces are zero, not the rounding of the common velocity, in every
form of the pair loops."""
import numpy as np
import pytest

import fsi_cases as fc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import Simulation  # noqa: E402

FORMS = {"cells": {}, "compact": dict(compact=1), "cell_rows": dict(rows=1), "tiles": dict(tile=1),
         "rows": dict(list=1)}


def _case(dim):
    if dim == 2:
        case = fc.floating_block(seed=1)
    else:
        case = fc.tiny_box_3d(seed=1)
        case.w_r, case.w_n = np.zeros((0, 3)), np.zeros((0, 3))
        case.gravity = (0.0, 0.0, 0.0)
        case.s_cons = np.zeros_like(case.s_cons)
        case.n_reinit = 0
        case.free_surface = 0
    v = np.array([3.0, 1.0, -2.0])[:dim]
    case.f_v = np.tile(v, (case.nf, 1))
    case.s_v0 = np.tile(v, (case.ns, 1))
    case.f_p = np.zeros(case.nf)
    return case


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("dim", [2, 3])
def test_a_common_velocity_leaves_no_density_rate(dim, form):
    sim = Simulation.from_case(_case(dim))
    sim.set_tuning(**{**dict(lanes=4, block=128, compact=0, tile=0, records=0, rows=0, list=0), **FORMS[form]})
    for _ in range(2):
        sim.step()
        sim.sync()
        g = sim.get_fluid()
        assert sim.info()["pairs_fs"] > 0
        assert not g["drho"].any() and not g["dvdt"].any()
    sim.close()
