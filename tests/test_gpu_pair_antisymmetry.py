"""The force of one fluid-solid pair on the fluid is the force on the solid with
the other sign, bit for bit: one fluid particle off the corner of a body with
exactly one solid particle in its support, at random distances, directions,
velocities, pressures and averaged solid motions, with the pair taken by the
fluid loops of every form."""
import numpy as np
import pytest

import fsi_cases as fc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import Simulation  # noqa: E402

FORMS = {"cells": {}, "compact": dict(compact=1), "cell_rows": dict(rows=1), "rows": dict(list=1)}
N = 48


def _case(dim, rng):
    """A body and one fluid particle with one body particle in its support."""
    case = fc.tiny_box(seed=1, with_walls=False) if dim == 2 else fc.tiny_box_3d(seed=1)
    if dim == 3:
        case.w_r, case.w_n = np.zeros((0, 3)), np.zeros((0, 3))
    case.n_reinit = 0
    corner = np.argmax(case.s_r0.sum(1))
    rc = 2 * 1.3 * case.f_dp
    while True:
        e = rng.uniform(0.15, 1.0, dim)
        x = case.s_r0[corner] + rc * rng.uniform(0.9, 0.999) * e / np.linalg.norm(e)
        if (np.linalg.norm(case.s_r0 - x, axis=1) < rc).sum() == 1:
            break
    case.f_r = x[None]
    case.f_v = rng.normal(0, 0.5, (1, dim))
    case.f_p = rng.uniform(-1, 1, 1) * case.f_rho0 * case.f_c0 ** 2 * 1e-2
    case.s_v0 = rng.normal(0, 0.5, case.s_r0.shape)
    return case


@pytest.mark.parametrize("form", list(FORMS))
@pytest.mark.parametrize("dim", [2, 3])
def test_one_pair_is_antisymmetric(dim, form):
    rng = np.random.default_rng(dim)
    cases = [_case(dim, rng) for _ in range(N)]
    sim = Simulation.from_cases(cases)
    sim.set_tuning(**{**dict(lanes=4, block=128, compact=0, tile=0, records=0, rows=0, list=0), **FORMS[form]})
    for b, case in enumerate(cases):
        sim.select(b).set_solid_state(abar=rng.normal(0, 20.0, case.s_r0.shape))
    sim.step(1e-6)
    sim.sync()
    for b in range(N):
        i = sim.select(b).info()
        assert i["pairs_fs"] == i["pairs_sf"] == 1
        f, s = np.asarray(i["mom_fs_fluid"])[:dim], np.asarray(i["mom_fs_solid"])[:dim]
        assert f.all() and np.array_equal(f, -s), (b, f, s)
    sim.close()
