"""Bodies around the windowed sub-step kernel's bounds against the FP64 oracle,
over two coarse steps of four sub-steps: a 3-D block whose windows fit shared
memory only with fewer particles per CTA than the sub-steps' share of the step
asks for, and the bodies of the cooperative kernel with a barrier per phase, a
3-D block whose windows fit at no size and a 2-D one of more particles per SM
than the windowed kernel holds.  The barrier kernel's waits that give up (limit
of one poll) are reported, and a restored checkpoint steps on bit for bit."""
import numpy as np
import pytest

import fsi_cases as fc
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import SphError, Simulation  # noqa: E402

TOL = 1e-5   # the bound of the other step-by-step comparisons
E_TIMEOUT = -6


def _block(n, dp=0.01, fluid=0):
    """A clamped block of n[0] x n[1] x n[2] particles in smooth motion; with
    `fluid` > 0 that many fluid particles per axis far from it, in the same context."""
    case = fc.tiny_box_3d(seed=1)
    none = np.zeros((0, 3))
    case.f_r, case.f_v, case.f_p, case.w_r, case.w_n = none, none, np.zeros(0), none, none
    hi = tuple(k * dp for k in n)
    x = case.s_r0 = fc.lattice((0, 0, 0), hi, dp)
    case.s_dp, case.f_dp = dp, 2 * dp
    case.s_v0 = np.stack([0.1 * np.sin(9 * x[:, 1]), 0.1 * np.cos(7 * x[:, 0]), 0.05 * np.sin(5 * x[:, 0] + 3 * x[:, 2])], 1)
    case.s_n0 = np.tile([1.0, 0.0, 0.0], (len(x), 1))
    case.s_cons = (x[:, 1] < 2 * dp).astype(np.uint8)
    case.s_v0[case.s_cons == 1] = 0.0
    case.domain_lo, case.domain_hi, case.tip = (-0.1,) * 3, tuple(h + 0.1 for h in hi), 0
    if fluid:
        lo = hi[0] + 0.5
        case.f_r = fc.lattice((lo, 0, 0), (lo + 2 * dp * fluid,) + (2 * dp * fluid,) * 2, 2 * dp)
        case.f_v, case.f_p = np.zeros_like(case.f_r), np.zeros(len(case.f_r))
        case.n_reinit = 0
        case.domain_hi = tuple(case.f_r.max(0) + 0.1)
    return case


CASES = {
    # 784 particles per layer: windows of 512 particles need 3.7k slots, of 166 3.4k; 232 KB hold 3.6k of them.
    # 32k fluid particles and one sub-step by the materials' estimate ask for 512.
    "window_smaller": lambda: _soft(_block((28, 28, 32), fluid=32)),
    # 1024 particles per layer: 4.1k slots at the least
    "barrier_3d": lambda: _block((32, 32, 34)),
    # 81k particles: more than 512 per SM
    "barrier_2d": lambda: _waves(fc.cantilever(L=1.0, t=1.0, dpS=1.0 / 283)),
}


def _soft(case):
    case.s_E = 1e-2
    return case


def _waves(case):
    """Velocities that vary over some ten particles, so that their FP32 rounding is small in the strains."""
    x, k = case.s_r0, 2 * np.pi / (16 * case.s_dp)
    case.s_v0 = 0.1 * np.stack([np.sin(k * x[:, 1]) * np.cos(k * x[:, 0]), np.cos(0.7 * k * x[:, 0])], 1)
    case.s_v0[case.s_cons == 1] = 0.0
    return case


@pytest.mark.parametrize("name", list(CASES))
def test_two_steps_against_the_oracle(name):
    case = CASES[name]()
    ref = O.OracleSim(case)
    _, _, dts = ref.suggest_dt()
    K, dt = 4, 3.9 * min(dts, 2e-3)
    sim = Simulation.from_case(case)
    sim.set_substeps(K)
    for _ in range(2):
        sim.step(dt)
        ref.step(dt, K)
    sim.sync()
    assert sim.info()["solid_path"] == 2
    s = sim.get_solid()
    I = np.eye(case.dim)
    for k, a, b in (("v", s["v"], ref.s_v), ("abar", s["abar"], ref.s_abar), ("vbar", s["vbar"], ref.s_vbar),
                    ("F-I", s["F"] - I, ref.s_F - I), ("dr", s["r"] - case.s_r0, ref.s_r - case.s_r0)):
        e = np.linalg.norm(a - b) / np.linalg.norm(b)
        print(name, k, f"{e:.1e}")
        assert e < TOL, (k, e)
    sim.close()


@pytest.mark.parametrize("name", ["barrier_3d", "barrier_2d"])
def test_a_barrier_that_gives_up_is_reported_and_a_checkpoint_recovers(name):
    case = CASES[name]()
    _, _, dts = O.OracleSim(case).suggest_dt()

    def make():
        sim = Simulation.from_case(case)
        sim.set_substeps(4)
        sim.step(3.9 * dts)
        sim.sync()
        return sim

    sim, other = make(), make()
    blob = sim.get_state()
    sim.set_wait_limit(1)
    for _ in range(3):
        sim.step(3.9 * dts)
    with pytest.raises(SphError) as e:
        sim.sync()
    assert e.value.code == E_TIMEOUT
    sim.set_wait_limit(0)
    sim.set_state(blob)
    for s in (sim, other):
        for _ in range(2):
            s.step(3.9 * dts)
        s.sync()
    a, b = sim.get_solid(), other.get_solid()
    for k in a:
        assert np.array_equal(a[k], b[k]), k
    sim.close()
    other.close()
