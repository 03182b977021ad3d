"""The instances of a batch take the pair-loop form, and a 3-D body the
sub-step arithmetic, that they take alone: a batch equals its instances
stepped alone to the last bit where its total would choose another form than
its members' sizes do, and where the members differ in form."""
import numpy as np
import pytest

import fsi_cases as fc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import Simulation  # noqa: E402


def _box(seed, n):
    return fc.tiny_box_3d(seed=seed, n=n, c0=40.0)


BATCHES = {
    # 40k particles in all, rows for none
    "channels_4x10k": lambda: [fc.channel_flag(seed=k) for k in range(4)],
    # rows for the second only (33k); the first slot is a cell-form instance's
    "mixed_2d": lambda: [fc.channel_flag(seed=1), fc.channel_flag(seed=2, dpF=0.1 / 18), fc.tiny_box(seed=3)],
    # rows for the first only (20k)
    "mixed_3d": lambda: [_box(1, (40, 8, 64)), _box(2, (10, 12, 8)), _box(3, (12, 8, 10))],
}


def _state(sim):
    out = {**{"f_" + k: v for k, v in sim.get_fluid().items()}, **{"s_" + k: v for k, v in sim.get_solid().items()}}
    info = sim.info()
    for k in ("t", "step", "last_dt", "last_K", "pairs_ff", "pairs_fw", "pairs_fs", "pairs_sf", "vmax_f", "vmax_s"):
        out[k] = np.asarray(info[k])
    return out


@pytest.mark.parametrize("cadence", [1, 3])
@pytest.mark.parametrize("name", list(BATCHES))
def test_batch_equals_its_instances_bitwise(name, cadence):
    cases = BATCHES[name]()
    for c in cases:
        c.n_reinit = 2
    stream = torch.cuda.Stream()
    batch = Simulation.from_cases(cases, stream=stream)
    batch.set_advection_cadence(cadence)
    batch.run(4, 0.0)
    blob = batch.get_state()          # inside an advection step where the cadence is 3
    batch.run(3, 0.0)
    batch.set_state(blob)
    batch.run(3, 0.0)
    batch.sync()
    for b, case in enumerate(cases):
        single = Simulation.from_case(case, stream=stream)
        single.set_advection_cadence(cadence)
        single.run(7, 0.0)
        single.sync()
        want, got = _state(single), _state(batch.select(b))
        for k in want:
            assert np.array_equal(got[k], want[k]), (b, k)
        single.close()
    batch.close()
