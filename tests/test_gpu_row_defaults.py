"""Neighbour rows where a context takes them by itself (32 768 fluid particles
in 2-D, 16 384 in 3-D), at every lane count, against the cell form that smaller
contexts use: both visit the same in-support pairs and differ in the order of
each particle's FP32 sums, so a step agrees to the per-step tolerance of the
pair loops (1e-5).  The dam break's many sub-steps start its solid branch before
the rows are built; its reinitialisation visits the cells."""
import numpy as np
import pytest

import fsi_cases as fc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import Simulation  # noqa: E402

TOL = 1e-5
CASES = {   # maker, rows by default, lanes by default
    "dam_4k": (lambda: fc.dam_gate(seed=3, dpF=1.8e-3), 0, 8),
    "dam_33k": (lambda: fc.dam_gate(seed=3, dpF=0.65e-3), 1, 2),
    "flag_10k": (lambda: fc.channel_flag(seed=3), 0, 8),
    "flag_33k": (lambda: fc.channel_flag(seed=3, dpF=0.1 / 18), 1, 2),
    "tank_15k": (lambda: fc.tiny_box_3d(seed=3, n=(31, 22, 22), c0=40.0), 0, 8),
    "tank_24k": (lambda: fc.tiny_box_3d(seed=3, n=(36, 26, 26), c0=40.0), 1, 4),
}


def rel(a, b):
    a, b = np.asarray(a, np.float64), np.asarray(b, np.float64)
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


def _step(case, tuning):
    sim = Simulation.from_case(case)
    if tuning:
        sim.set_tuning(**tuning)
    t = sim.tuning()
    sim.step()   # the first step reinitialises the density
    sim.sync()
    out = t, sim.get_fluid(), sim.get_solid(), sim.info()
    sim.close()
    return out


@pytest.mark.parametrize("name", list(CASES))
def test_default_rows_and_every_lane_count_against_the_cell_form(name):
    make, list_on, lanes = CASES[name]
    case = make()
    case.n_reinit = 1
    t, *default = _step(case, None)
    assert (t["list"], t["lanes"]) == (list_on, lanes)
    _, gc, sc, ic = _step(case, dict(lanes=4, block=128, compact=0, rows=0, list=0))
    rows = [_step(case, dict(lanes=k, block=128, compact=0, rows=0, list=1))[1:]
            for k in ((2, 4, 8) if case.dim == 2 else (4, 8, 16))]
    for g, s, i in [default] + rows:
        e = {k: rel(g[k], gc[k]) for k in ("dvdt", "drho", "v", "rho")}
        if case.ns:
            e["fF"], e["v_s"] = rel(s["fF"], sc["fF"]), rel(s["v"], sc["v"])
        print(name, {k: f"{v:.1e}" for k, v in e.items()})
        assert max(e.values()) < TOL, e
        for k in ("pairs_ff", "pairs_fw", "pairs_fs", "pairs_sf"):
            assert i[k] == ic[k], k
