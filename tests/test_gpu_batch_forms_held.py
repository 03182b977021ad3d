"""A batch whose instances differ in the form of the pair loops, inside an
advection step: one form set for all there (by the caller or by the
autotuner), and a checkpoint taken there and restored into a batch with rows
for all, get the missing instances' rows and hold the configuration on like the
batch that was left alone."""
import numpy as np
import pytest

import fsi_cases as fc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import Simulation  # noqa: E402

TOL = 1e-5   # the two forms' per-step tolerance (the order of FP32 sums)
BATCHES = {   # rows for the first, for the second instance
    "3d": lambda: [fc.tiny_box_3d(seed=1, n=(40, 8, 64), c0=40.0), fc.tiny_box_3d(seed=2, n=(10, 12, 8), c0=40.0)],
    "2d": lambda: [fc.channel_flag(seed=1), fc.channel_flag(seed=2, dpF=0.1 / 18)],
}


@pytest.mark.parametrize("how", ["tuning", "autotune", "checkpoint"])
@pytest.mark.parametrize("name", list(BATCHES))
def test_one_form_for_all_inside_an_advection_step(name, how):
    cases = BATCHES[name]()
    stream = torch.cuda.Stream()
    alone, other = Simulation.from_cases(cases, stream=stream), Simulation.from_cases(cases, stream=stream)
    assert alone.tuning()["list"] == 1
    rows = dict(lanes=4, block=128, compact=0, rows=0, list=1)
    if how == "checkpoint":
        other.set_tuning(**rows)
    for sim in (alone, other):
        sim.set_advection_cadence(8)
        sim.run(3, 0.0)
        sim.sync()
    if how == "tuning":
        other.set_tuning(**rows)
    elif how == "autotune":
        other.autotune(0.0, steps=6)
    else:
        other.set_state(alone.get_state())
    for _ in range(3):
        for sim in (alone, other):
            sim.run(1, 0.0)
            sim.sync()
        for b in range(len(cases)):
            x, y = alone.select(b).get_fluid(), other.select(b).get_fluid()
            for k in ("dvdt", "drho", "v"):
                e = np.linalg.norm(x[k].astype(np.float64) - y[k]) / np.linalg.norm(x[k].astype(np.float64))
                assert e < TOL, (b, k, e)
    alone.close()
    other.close()
