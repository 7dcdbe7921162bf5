"""The read-back kernels: the wide moments of the FP32 distributions against FP64
sums of the exported PDFs."""
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


@pytest.mark.parametrize("precision", ["fp64", "fp32", "f16s", "bf16s"])
@pytest.mark.parametrize("dims", [(13, 11, 17), (32, 24, 20)])
def test_exported_density_and_velocity_are_the_moments_of_the_exported_pdfs(fsl, precision, dims):
    """rho = sum f and u = sum c f / rho of the PDFs exported beside them, in
    FP64: a reference sum of 19 terms rounds by at most 18 halves of an ulp of
    the sum of their magnitudes, the quotient by one more.  Cells that never
    held liquid (all PDFs zero in FP32 storage) read 0."""
    sc = S.random_bubbles(*dims, n_bubbles=3, r_min=2.5, r_max=4.0, u_max=0.05, sigma=4e-3, seed=2)
    sim = fsl.Simulation.from_scenarios([sc], precision=precision)
    for steps in (0, 7):
        sim.step(steps)
        g = sim.fields(0, ("rho", "u", "pdf"))
        f = g["pdf"]
        rho, u = macro(f)
        zero = (f == 0.0).all(0)
        eps = 2.0 ** -53
        tol = 18 * eps * np.abs(f).sum(0)
        assert np.all(g["rho"][zero] == 0.0) and np.all(g["u"][:, zero] == 0.0)
        live = ~zero
        assert np.all(np.abs(g["rho"] - rho)[live] <= tol[live])
        bound = (2 * tol + tol * np.abs(u) + 4 * eps * np.abs(u) * rho) / np.where(zero, 1.0, rho)
        assert np.all((np.abs(g["u"] - u) <= bound)[:, live])
    sim.close()
