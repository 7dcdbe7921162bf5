"""Liquid lattices with an odd number of cells in 16-bit storage, whose last cell has
padding for a partner in its pair, against FP64: thin ones, ones with walls, alone and
as the last domain of a batch."""
import numpy as np
import pytest

from paper_1604_01632_gb300 import scenarios as S

pytestmark = pytest.mark.gpu
STEPS = 6


@pytest.fixture(scope="module")
def fsl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_01632_gb300 import build, fsl as F
    build.build()
    return F


def run(fsl, shapes, walls, precision, form):
    par = [dict(nx=nx, ny=ny, nz=nz, collision=1, tau=0.8) for nx, ny, nz in shapes]
    sim = fsl.Simulation(par, precision=precision)
    for d, (nx, ny, nz) in enumerate(shapes):
        z, y, x = np.ogrid[:nz, :ny, :nx]
        flags = np.full((nz, ny, nx), S.LIQUID, dtype=np.uint8)
        if walls:
            flags[:, 0] = S.OBSTACLE
        wave = 0.02 * np.sin(2 * np.pi * (x / nx + 2 * y / ny + z / nz))
        u = np.stack([wave, 0.7 * wave, -0.5 * wave]).reshape(-1)
        sim.init_geometry(d, flags.reshape(-1), np.ones(flags.size), np.ones(flags.size), u)
    sim.set_stream_form(form)
    sim.step(STEPS)
    out = [sim.fields(d, ("flags", "pdf")) for d in range(len(shapes))]
    sim.close()
    return out


@pytest.mark.parametrize("precision, digits", [("f16s", 11), ("bf16s", 8)])
@pytest.mark.parametrize("form", [0, 2, 5, 7])
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shapes", [[(5, 7, 1)], [(255, 3, 1)], [(33, 31, 1)], [(1, 3, 5)], [(21, 33, 7)],
                                    [(16, 16, 4), (31, 9, 1)]])
def test_last_cell_of_an_odd_lattice(fsl, shapes, walls, form, precision, digits):
    ref = run(fsl, shapes, walls, "fp64", 0)
    got = run(fsl, shapes, walls, precision, form)
    # a stored deviation is off by half a unit in the last place, 2^-digits of it at
    # most; a step of the collision hands on no more than the sum over the directions
    # of what it is given, and the deviations stay below 3 w_a |c u| < 0.03
    bound = (STEPS + 1) * 19 * 0.03 * 2.0 ** -digits
    for a, b in zip(ref, got):
        assert np.array_equal(a["flags"], b["flags"])
        assert np.abs(a["pdf"] - b["pdf"]).max() < bound
