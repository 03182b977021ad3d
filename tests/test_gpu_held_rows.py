"""Neighbour rows with a held pair configuration: a checkpoint taken inside an
advection step continues bit for bit, in the same context after it stepped on
and in a fresh one; autotuning inside one leaves the rest of it as it was; and
where the held configuration has no rows (the form was changed, or the
checkpoint came from a context without), they are built from it and it is held
on, as the cell form does."""
import numpy as np
import pytest

import fsi_cases as fc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import Simulation  # noqa: E402

TOL = 1e-5   # the two forms' per-step tolerance (the order of FP32 sums)
CASES = {
    "channel_flag": lambda: fc.channel_flag(seed=2),
    "tiny_box_3d": lambda: fc.tiny_box_3d(seed=2),
    "tank_24k": lambda: fc.tiny_box_3d(seed=3, n=(36, 26, 26), c0=40.0),   # rows by default
}


def _sim(case, list_on, cadence):
    sim = Simulation.from_case(case, stream=torch.cuda.Stream())
    sim.set_tuning(4, 128, compact=0, rows=0, list=list_on)
    sim.set_advection_cadence(cadence)
    return sim


def _steps(sim, n):
    for _ in range(n):
        sim.step()
    sim.sync()


def _state(sim):
    return {**{"f_" + k: v for k, v in sim.get_fluid().items()}, **{"s_" + k: v for k, v in sim.get_solid().items()}}


def _same(a, b, what):
    for k in a:
        assert np.array_equal(a[k], b[k]), (what, k)


def _close(a, b, what):
    for k in ("f_dvdt", "f_drho", "f_v", "s_fF"):
        x, y = a[k].astype(np.float64), b[k].astype(np.float64)
        assert np.linalg.norm(x - y) < TOL * np.linalg.norm(y), (what, k, np.linalg.norm(x - y) / np.linalg.norm(y))


@pytest.mark.parametrize("cadence", [4, "auto"])
@pytest.mark.parametrize("name", list(CASES))
def test_checkpoint_inside_an_advection_step_continues_bitwise(name, cadence):
    case = CASES[name]()
    sim = _sim(case, 1, cadence)
    _steps(sim, 6)
    blob = sim.get_state()
    _steps(sim, 3)
    want = _state(sim)
    _steps(sim, 2)                 # past a rebuild: other rows and other lists
    sim.set_state(blob)
    _steps(sim, 3)
    _same(_state(sim), want, "same context")
    fresh = _sim(case, 1, cadence)
    fresh.set_state(blob)
    _steps(fresh, 3)
    _same(_state(fresh), want, "fresh context")
    sim.close()
    fresh.close()


@pytest.mark.parametrize("name", list(CASES))
def test_autotune_inside_an_advection_step_keeps_the_rest_of_it(name):
    case = CASES[name]()
    a, b = _sim(case, 1, 8), _sim(case, 1, 8)
    for sim in (a, b):
        _steps(sim, 3)
    a.autotune(0.0, steps=6)       # trials go past the next rebuild
    for sim in (a, b):
        _steps(sim, 1)
    _close(_state(a), _state(b), "autotune")
    a.close()
    b.close()


@pytest.mark.parametrize("how", ["tuning", "checkpoint"])
@pytest.mark.parametrize("name", list(CASES))
def test_a_held_configuration_without_rows_gets_them(name, how):
    case = CASES[name]()
    cells, other = _sim(case, 0, 8), _sim(case, 0 if how == "tuning" else 1, 8)
    for sim in (cells, other):
        _steps(sim, 3)
    if how == "tuning":
        other.set_tuning(4, 128, compact=0, rows=0, list=1)
    else:
        other.set_state(cells.get_state())
    for _ in range(3):               # the rest of the advection step
        for sim in (cells, other):
            _steps(sim, 1)
        _close(_state(other), _state(cells), how)
    cells.close()
    other.close()
