"""The number-density sums of the reinitialisation against 64 bits.  A lattice
whose particles are off by 1e-7 of the spacing has densities that deviate from
rho0 by about 1e-7, so the FP32 number they end in resolves 1e-14 and the pair
sums themselves are seen.

Bound: a pair's shape is good to 1e-14 rms (the arithmetic's errors restated in
extended precision), a particle has at most 80 pairs and the shapes sum to
more than 3 with its own, so the sum's relative error is below 80 * 1e-14 / 3
= 2.7e-13 if all errors of a particle agreed in sign; asked for the rms over
the particles."""
import numpy as np
import pytest

import fsi_cases as fc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_1911_13255_gb300 import Simulation  # noqa: E402

TOL = 2.7e-13


def _case(dim, n, dp):
    case = fc.tiny_box(seed=1) if dim == 2 else fc.tiny_box_3d(seed=1)
    hi = (n * dp,) * dim
    case.f_r = fc.jitter(fc.lattice((0.0,) * dim, hi, dp), dp, 1e-7, np.random.default_rng(3))
    case.f_v, case.f_p = np.zeros_like(case.f_r), np.zeros(len(case.f_r))
    case.f_dp = dp
    none = np.zeros((0, dim))
    case.w_r, case.w_n, case.s_r0, case.s_v0, case.s_n0 = none, none, none, none, none
    case.s_cons = np.zeros(0, np.uint8)
    case.gravity = (0.0, 0.0, 0.0)
    case.domain_lo = tuple([-dp] * dim + [0.0] * (3 - dim))
    case.domain_hi = tuple([n * dp + dp] * dim + [0.0] * (3 - dim))
    case.free_surface, case.n_reinit = 0, 1
    return case


def _shape(r, h):
    q = r / h
    return np.where(q < 2, (1 - 0.5 * q) ** 4 * (1 + 2 * q), 0.0)


@pytest.mark.parametrize("rows", [0, 1])
@pytest.mark.parametrize("dim,n,dp", [(2, 40, 0.01), (2, 37, 0.00093), (3, 18, 0.02), (3, 16, 0.0137)])
def test_density_sums_against_64_bits(dim, n, dp, rows):
    case = _case(dim, n, dp)
    h, r = 1.3 * dp, case.f_r
    inner = np.flatnonzero(np.all((r > 2.1 * h) & (r < n * dp - 2.1 * h), axis=1))
    assert len(inner) > 50
    m = int(np.ceil(2 * h / dp)) + 1
    g = np.stack(np.meshgrid(*[np.arange(-m, m + 1) * dp] * dim), -1).reshape(-1, dim)
    sigma0 = _shape(np.linalg.norm(g, axis=1), h).sum()
    want = np.array([_shape(np.linalg.norm(r - r[i], axis=1), h).sum() for i in inner]) / sigma0 - 1
    assert 1e-9 < np.abs(want).max() < 1e-5
    sim = Simulation.from_case(case)
    sim.set_tuning(4, 128, compact=0, rows=0, list=rows)
    sim.step(1e-13)
    sim.sync()
    got = sim.get_fluid()["rho"][inner] / case.f_rho0 - 1
    err = np.sqrt(np.mean((got - want) ** 2))
    print(dim, n, rows, f"{err:.2e}", f"{np.abs(got - want).max():.2e}")
    assert err < TOL, err
    sim.close()
