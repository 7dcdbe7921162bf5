"""Read-back of FP32 distributions that nearly cancel: density and velocity are those
of FP64 sums and divisions, also where a distribution is close to zero or the momentum
is small against its terms."""
import numpy as np
import pytest

from paper_1604_01632_gb300 import scenarios as S

from parity_util import macro

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fsl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_01632_gb300 import build, fsl as F
    build.build()
    return F


def velocities(kind, n):
    rng = np.random.Generator(np.random.PCG64(7))
    if kind == "rest":
        return 1e-9 * rng.standard_normal((3, n))
    if kind == "fast":
        return rng.uniform(-0.4, 0.4, (3, n))
    # u_x = u_y at the root of 1 - 3 u + 1.5 u^2: f_eq of direction -x is nearly zero
    root = 1.0 - 1.0 / np.sqrt(3.0)
    return np.stack([root + 1e-6 * rng.standard_normal(n), root + 1e-6 * rng.standard_normal(n),
                     1e-7 * rng.standard_normal(n)])


@pytest.mark.parametrize("precision", ["fp32", "f16s", "bf16s"])
@pytest.mark.parametrize("kind", ["rest", "fast", "near zero"])
def test_density_and_velocity_are_those_of_fp64(fsl, kind, precision):
    """The FP64 sums of FP32 terms that span less than 2^29 are exact, so the density
    is equal; a quotient rounds once, so the velocity is the neighbouring value at most.
    (Terms further apart, which "near zero" has a few of, add an ulp of the sum each.)"""
    nx, ny, nz = 64, 48, 32
    n = nx * ny * nz
    sim = fsl.Simulation([dict(nx=nx, ny=ny, nz=nz)], precision=precision)
    sim.init_geometry(0, np.full(n, S.LIQUID, dtype=np.uint8), np.ones(n), np.ones(n), velocities(kind, n).reshape(-1))
    g = sim.fields(0, ("rho", "u", "pdf"))
    sim.close()
    f = g["pdf"].reshape(19, n)
    rho, u = macro(f)
    rho, u = rho.reshape(n), u.reshape(3, n)
    least = np.abs(f).min(0)
    exact = np.abs(f).max(0) < 2.0 ** 24 * least
    assert exact.mean() > 0.5   # the comparison covers most cells
    assert np.array_equal(g["rho"].reshape(n)[exact], rho[exact])
    assert np.all(np.abs(g["u"].reshape(3, n) - u)[:, exact] <= np.spacing(np.abs(u))[:, exact])
    tol = 19 * 2.0 ** -53 * np.abs(f).sum(0)
    assert np.all(np.abs(g["rho"].reshape(n) - rho) <= tol)
    assert np.all(np.abs(g["u"].reshape(3, n) - u) <= 4 * tol / rho)
