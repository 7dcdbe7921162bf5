"""Steps whose interface kernel forms the fill levels (the two-kernel form with
the list in cell order, the tile-fused forms): pooled excess mass, and the
interface list when forms change."""
import numpy as np
import pytest

from paper_1604_01632_gb300 import scenarios as S

from parity_util import compare_exact, gpu_state, oracle_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fsl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_01632_gb300 import build, fsl as F
    build.build()
    return F


def _with_lone_cells(seed):
    """Moving bubbles and a few interface cells alone in the liquid: each fills at
    once (it separates nothing), has no interface neighbour to take its excess
    mass, and so feeds the pool that every interface cell shares."""
    sc = S.random_bubbles(26, 22, 20, n_bubbles=4, r_min=2.5, r_max=4.5, u_max=0.05, sigma=4e-3, seed=seed)
    rng = np.random.Generator(np.random.PCG64(seed))
    liq = sc.flags == S.LIQUID
    free = liq.copy()
    for dz in (-2, -1, 0, 1, 2):
        for dy in (-2, -1, 0, 1, 2):
            for dx in (-2, -1, 0, 1, 2):
                free &= np.roll(liq, (dz, dy, dx), (0, 1, 2))
    at = np.argwhere(free)
    for z, y, x in at[rng.permutation(len(at))[:3]]:
        sc.flags[z, y, x] = S.INTERFACE
        sc.fill[z, y, x] = rng.uniform(0.2, 0.8)
    return sc


@pytest.mark.parametrize("form,order", [(5, 1), (5, 0), (0, 0)])
def test_pooled_excess_mass_bitexact(fsl, oracle_mod, form, order):
    scs = [_with_lone_cells(s) for s in (0, 1)]
    sim = fsl.Simulation.from_scenarios(scs, precision="fp64")
    sim.set_interface_order(order)
    sim.set_stream_form(form)
    oras = [oracle_mod.Oracle.from_scenario(s) for s in scs]
    pooled = 0
    prev = 0
    for k in (1, 2, 3, 12):
        sim.step(k - prev)
        for o in oras:
            before = o.flags()
            o.step(k - prev)
            pooled += int(((before == S.INTERFACE) & (o.flags() == S.LIQUID)).sum())
        prev = k
        for d, o in enumerate(oras):
            compare_exact(gpu_state(sim, d), oracle_state(o), what=f"form {form} order {order} domain {d} step {k}")
    assert pooled >= 3
    sim.close()


def test_switching_forms_keeps_the_interface_list(fsl):
    """The tile-fused forms keep no interface list; a form that needs one gets it
    rebuilt, in cell order: an FP32 handle that goes 7 -> 5 -> 7 -> 4 follows the
    split form within rounding."""
    sc = S.random_bubbles(40, 36, 33, n_bubbles=8, r_min=3.0, r_max=6.0, u_max=0.05, sigma=4e-3, seed=4)
    ref = fsl.Simulation.from_scenarios([sc], precision="fp32")
    ref.set_stream_form(0)
    ref.step(24)
    sim = fsl.Simulation.from_scenarios([sc], precision="fp32")
    for form in (7, 5, 7, 4):
        if form == 4:
            sim.set_interface_order(1)
        sim.set_stream_form(form)
        sim.step(6)
    a, b = ref.fields(0, ("flags", "fill")), sim.fields(0, ("flags", "fill"))
    assert np.mean(a["flags"] == b["flags"]) > 0.999
    assert np.linalg.norm(a["fill"] - b["fill"]) / np.linalg.norm(a["fill"]) < 1e-4
    assert abs(ref.total_mass() / sim.total_mass() - 1.0) < 1e-5
    ref.close()
    sim.close()
