"""3-D bodies of up to one cluster's size take the windowed sub-step kernel alone
(above 512 particles) and the cluster kernel in a batch.  Both give the same
bits: path against path at body sizes around the CTAs' bounds of either kernel,
and a batch against its instances alone."""
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


def _plate(rows):
    """A box of `rows` fluid particles in height; its plate takes 60 % of that."""
    return _box(5, (10, rows, 8))


def _state(sim):
    out = {**{"f_" + k: v for k, v in sim.get_fluid().items()}, **{"s_" + k: v for k, v in sim.get_solid().items()}}
    info = sim.info()
    for k in ("t", "step", "last_dt", "last_K", "vmax_f", "vmax_s", "amax_s"):
        out[k] = np.asarray(info[k])
    return out


@pytest.mark.parametrize("rows", [6, 8, 12, 14, 20, 36, 52])
@pytest.mark.parametrize("stiff", [1.0, 400.0])
def test_window_and_cluster_kernels_agree_bitwise(rows, stiff):
    """stiff: more sub-steps, and with them other numbers of particles per CTA of the window plan."""
    case = _plate(rows)
    case.s_E *= stiff
    states = []
    for path in (1, 2):
        sim = Simulation.from_case(case)
        sim.set_solid_path(path)
        for _ in range(4):
            sim.step()
        sim.sync()
        assert sim.info()["solid_path"] == path
        states.append(_state(sim))
        sim.close()
    assert np.abs(states[0]["s_abar"]).max() > 0
    for k in states[0]:
        assert np.array_equal(states[0][k], states[1][k]), k


def test_batch_with_large_plates_equals_its_instances_bitwise():
    cases = [_box(1, (10, 36, 8)), _box(2, (24, 40, 24)), _box(3, (10, 12, 8)), _box(4, (12, 22, 10))]
    assert sorted(c.ns for c in cases)[-3] > 512
    stream = torch.cuda.Stream()
    batch = Simulation.from_cases(cases, stream=stream)
    batch.run(6, 0.0)
    batch.sync()
    for b, case in enumerate(cases):
        single = Simulation.from_case(case, stream=stream)
        single.run(6, 0.0)
        single.sync()
        want, got = _state(single), _state(batch.select(b))
        for k in want:
            assert np.array_equal(got[k], want[k]), (b, k)
        single.close()
    batch.close()
