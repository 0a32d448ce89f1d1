"""The Poisson solves in units far from 1 (float ranges, not the scheme): the potential is
linear in G, in rho and in h^2, so a solve whose constants or densities come near the ends of
the float range has the potential of a solve in mid-range units, scaled."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from oracle import poisson  # noqa: E402
from paper_1607_01105_gb300 import ppml  # noqa: E402

pytestmark = pytest.mark.gpu

F32 = ppml.PPML_F32
O, P = ppml.OUTFLOW, ppml.PERIODIC
TOL = 2e-5  # the FP32 solves' bar, of the largest potential
CGS = 6.674e-8  # G in cm^3 g^-1 s^-2


def _density(n):
    x, y, z = [np.arange(m) / m for m in n]
    z, y, x = np.meshgrid(z, y, x, indexing="ij")
    return 1.0 + 0.5 * np.sin(2 * np.pi * x) * np.cos(2 * np.pi * y) + 0.2 * np.cos(4 * np.pi * z)


def _solve(n, h, rho, G, isolated, printed=False):
    u = [torch.ones(int(np.prod(n)), device="cuda") for _ in range(6)]
    grid = ppml.Grid(n, (h,) * 3, 1.4, 0.2, (O if isolated else P,) * 6, F32, u0=u)
    r = torch.as_tensor(rho.ravel()).to("cuda", torch.float32)
    phi = torch.empty_like(r)
    if isolated:
        grid.poisson_isolated(r, phi, G, printed_rhs=printed)
    else:
        grid.poisson_periodic(r, phi, G)
    return r.double().cpu().numpy().reshape(rho.shape), phi.double().cpu().numpy().reshape(rho.shape)


# (cell size, density scale, G): 30 Mpc and 30 Gpc cells in CGS units (coefficients of 1e39 and
# more), SI ones, a tiny constant with a large density, and units of order 1
UNITS = [(1e23, 1e-24, CGS), (1e26, 1e-30, CGS), (1e29, 1e-34, CGS), (1e24, 1e-26, 6.674e-11),
         (1e-18, 1e30, 1e-8), (0.03, 1.0, 1.7)]


@pytest.mark.parametrize("h,scale,G", UNITS)
@pytest.mark.parametrize("n", [(32, 24, 20), (64, 64, 64)])
def test_periodic_potential_in_any_units(n, h, scale, G):
    rho, got = _solve(n, h, scale * _density(n), G, False)
    ref = poisson.solve_periodic(rho, h, G)
    assert np.all(np.isfinite(got))
    assert np.max(np.abs(got - ref)) <= TOL * np.max(np.abs(ref))


def _blob(n):
    x, y, z = [(np.arange(m) + 0.5) / m - 0.5 for m in n]
    z, y, x = np.meshgrid(z, y, x, indexing="ij")
    return np.exp(-(x * x + 1.5 * (y - 0.1) ** 2 + 2.0 * (z + 0.05) ** 2) / 0.05)


# grids of the dense transforms and of the transforms of the odd extension
@pytest.mark.parametrize("n", [(20, 24, 28), (300, 12, 10)])
@pytest.mark.parametrize("printed", [False, True])
@pytest.mark.parametrize("h,scale,G", UNITS)
def test_isolated_potential_in_any_units(n, printed, h, scale, G):
    rho, got = _solve(n, h, scale * _blob(n), G, True, printed)
    ref = poisson.solve_isolated(rho, h, G, printed_rhs=printed)
    assert np.all(np.isfinite(got))
    assert np.max(np.abs(got - ref)) <= TOL * np.max(np.abs(ref))


# densities near the ends of the float range: second moments and neighbour sums beyond it,
# products' errors below it
@pytest.mark.parametrize("n", [(64, 64, 48), (300, 20, 12), (20, 40, 41)])
@pytest.mark.parametrize("scale,G", [(3e38, 1e-23), (1e37, 1e-20), (1e35, 1e-37), (1e-37, 1e25)])
def test_isolated_potential_of_any_density(n, scale, G):
    rho, got = _solve(n, 0.03, scale * _blob(n), G, True)
    ref = poisson.solve_isolated(rho, 0.03, G)
    assert np.all(np.isfinite(got))
    assert np.max(np.abs(got - ref)) <= TOL * np.max(np.abs(ref))
