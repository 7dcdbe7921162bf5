"""The two-kernel form runs as one tile-fused kernel from 2^20 cells on in the
FP32-collide storage forms: its states are those of the separate kernels (form 8
keeps them), and the two tile sizes agree.  Both kernels round every operation of a
rebuilt PDF in the same, written-out way, so the comparison is bit for bit."""
import numpy as np
import pytest

from paper_1604_01632_gb300 import scenarios as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fsl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_01632_gb300 import build, fsl as F
    build.build()
    return F


# 1,061,208 cells; rows of odd length; a batch whose domains add up to 2^20
SHAPES = {"one": [(102, 102, 102)], "odd rows": [(101, 103, 105)], "batch": [(88, 80, 75), (64, 96, 90)]}


@pytest.mark.parametrize("precision", ["fp32", "f16s", "bf16s"])
@pytest.mark.parametrize("shape", list(SHAPES))
def test_same_state_as_the_separate_kernels(fsl, shape, precision):
    scs = [S.random_bubbles(*dims, n_bubbles=40, r_min=4.0, r_max=9.0, u_max=0.08, sigma=4e-3, seed=d)
           for d, dims in enumerate(SHAPES[shape])]
    state = {}
    for form in (5, 8, 6, 7):
        sim = fsl.Simulation.from_scenarios(scs, precision=precision)
        sim.set_interface_order(1)
        sim.set_stream_form(form)
        sim.step(12)
        state[form] = [sim.fields(d, ("flags", "fill", "mass", "pdf")) for d in range(len(scs))]
        sim.close()
    for a, b in ((5, 8), (6, 7)):
        for d, (x, y) in enumerate(zip(state[a], state[b])):
            for name in x:
                assert np.array_equal(x[name], y[name]), f"forms {a} and {b}, domain {d}, {name}"
