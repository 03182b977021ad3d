"""The windowed sub-step kernel (one body over a grid of CTAs that exchange
the particles of their windows) against the FP64 oracle: bodies that end
inside a CTA, on its boundary and one particle past it, of a few CTAs and of
more than one wait set, in 2-D (chosen by the grid path) and in 3-D (chosen by
size), over two coarse steps of several sub-steps."""
import numpy as np
import pytest

import fsi_cases as fc
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import Simulation  # noqa: E402

TOL = 1e-5   # the bound of the other step-by-step comparisons (per-step accelerations, relative L2)


def _beam(columns, rows, dp=0.005):
    """A clamped beam of (columns + 4) x rows particles, no fluid."""
    return fc.cantilever(L=columns * dp, t=rows * dp, dpS=dp)


CASES = {
    "beam_32": (lambda: _beam(12, 2), 2),          # exactly one CTA's particles
    "beam_33": (lambda: _beam(7, 3), 2),           # one particle in the second CTA
    "gate_2mm": (lambda: fc.dam_gate(seed=1, dpF=2e-3), 2),
    "gate_half_mm": (lambda: fc.dam_gate(seed=1, dpF=5e-4), 0),      # beyond one cluster: 6400 particles
    "plate_448": (lambda: fc.tiny_box_3d(seed=2, n=(10, 12, 8)), 2),
    "plate_1408": (lambda: fc.tiny_box_3d(seed=2, n=(10, 36, 8)), 2),
    "plate_2304": (lambda: fc.tiny_box_3d(seed=2, n=(10, 60, 8)), 0),
}



@pytest.mark.parametrize("name", list(CASES))
def test_two_steps_against_the_oracle(name):
    make, path = CASES[name]
    case = make()
    ref = O.OracleSim(case)
    _, _, dts = ref.suggest_dt()
    K = 5
    dt = 4.9 * dts if case.nf == 0 else min(4.9 * dts, ref.suggest_dt()[0])
    sim = Simulation.from_case(case)
    sim.set_solid_path(path)
    sim.set_substeps(K)
    for _ in range(2):
        sim.step(dt)
        ref.step(dt, K)
    sim.sync()
    assert sim.info()["solid_path"] == 2
    s = sim.get_solid()
    I = np.eye(case.dim)
    # a body that only falls with the water around it moves rigidly for its
    # first steps: F - I and the displacement then compare against the size
    # that one velocity rounding makes over the step
    for k, a, b, floor in (("v", s["v"], ref.s_v, 0.0), ("abar", s["abar"], ref.s_abar, 0.0),
                           ("vbar", s["vbar"], ref.s_vbar, 0.0),
                           ("F-I", s["F"] - I, ref.s_F - I, 2.0 ** -24 * np.sqrt(case.ns)),
                           ("dr", s["r"] - case.s_r0, ref.s_r - case.s_r0, 0.0)):
        e = np.linalg.norm(a - b)
        assert e <= TOL * np.linalg.norm(b) + floor, (name, k, e, np.linalg.norm(b))
    sim.close()
