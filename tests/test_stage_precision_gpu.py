"""One step of the FP64 form's three-dimensional stage against extended precision, below the rounding
that the parity tests resolve.  The filter is taken out by its own coefficient: at the largest alpha_f
below 1/2 its increment, (1 - 2 alpha) delta^10 f / 1024, is 1e-16 of delta^10 f."""
import numpy as np
import pytest

from paper_2506_03027_gb300 import cfs
from paper_2506_03027_gb300 import inputs as I

from extended import step
from gpu_util import ensure_built

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    ensure_built()


def flow(c, seed):
    """A smooth periodic flow with velocities and a pressure disturbance of about 1."""
    rng = np.random.default_rng(seed)
    z, y, x = np.meshgrid(*[2 * np.pi * np.arange(n) / n for n in (c.nz, c.ny, c.nx)], indexing="ij")

    def wave():
        return np.sin(x * rng.integers(-2, 3) + y * rng.integers(-2, 3) + z * rng.integers(-2, 3) + rng.uniform(0, 2 * np.pi))
    rho = 1 + 0.3 * c.mach ** 2 * wave()
    u = [0.6 * wave() + 0.3 * wave() for _ in range(3)]
    U = np.empty((5, c.nz, c.ny, c.nx))
    U[0] = rho
    for a in range(3):
        U[1 + a] = rho * u[a]
    U[4] = (1 / (c.gamma * c.mach ** 2) + 0.3 * wave()) / (c.gamma - 1) + 0.5 * rho * sum(v * v for v in u)
    return U


FORMS = {"viscous": {}, "power_law": {"visc_law": 1}, "euler": {"viscous": False}, "compact": {"viscous": False, "compact": 1},
         "order2": {"order": 2}}
_steps = {}


def one_step(form, mach):
    """(case, state and error after one step at a CFL number of 0.5), each computed once."""
    if (form, mach) not in _steps:
        c = I.tgv_case(20, 1, "SA").replace(mach=mach, alpha_f=float(np.nextafter(0.5, 0)), **FORMS[form])
        c = c.replace(dt=0.5 * c.dx / 3 / (1 + 1 / mach))
        U0 = flow(c, 3)
        s = cfs.Solver(c)
        s.set_schedule()
        s.set_state(U0)
        s.step(1)
        U = s.get_state()
        s.close()
        _steps[form, mach] = c, U, (U - step(c, U0)).astype(np.float64)
    return _steps[form, mach]


def rms(x):
    return float(np.sqrt(np.mean(np.square(x))))


def rounding(c, U, v):
    """The rounding of a variable by the sums U + B Q of a step's stages."""
    return np.sqrt(c.stages) * rms(np.spacing(np.abs(U[v])) / np.sqrt(12))


# the pressure comes from rho E, 179 at M = 0.1 and 17,857 at M = 0.01, against a dynamic one of about 1
@pytest.mark.parametrize("mach", [0.1, 0.01])
@pytest.mark.parametrize("form", list(FORMS))
def test_momentum_of_one_step(form, mach):
    c, U, e = one_step(form, mach)
    # a difference has at most twice a flux's error per spacing and there are three axes, each of
    # independent errors; a flux holds (gamma - 1) times the rounding of the stage's rho E, and two
    # roundings to 2^-48 of fluxes and energy deviations of about 1.5
    flux = (c.gamma - 1) * rounding(c, U, 4) + 2 * 2.0 ** -48 * 1.5
    tol = 2 * np.sqrt(3) * c.dt / c.dx * flux
    for v in (1, 2, 3):
        assert rms(e[v]) <= rounding(c, U, v) + tol, (v, rms(e[v]), rounding(c, U, v), tol)


# the mass flux is the momentum, the energy flux 250 times it at M = 0.1
@pytest.mark.parametrize("mach", [0.1, 0.01])
@pytest.mark.parametrize("form", list(FORMS))
def test_density_and_energy_of_one_step(form, mach):
    c, U, e = one_step(form, mach)
    # the rounding of the sums U + B Q, and what else there is, independent of it, below half of that:
    # sqrt(1 + 1/4)
    for v in (0, 4):
        assert rms(e[v]) <= 1.12 * rounding(c, U, v), (v, rms(e[v]), rounding(c, U, v))
