"""The paper's split trigger (split_trigger = 1) decides on the fill levels of the
start of the step in every stream-collide form, so the forms that form the new fill
levels in the interface kernel (the tile-fused ones, and the two-kernel ones with the
interface list in cell order) relabel the same bubbles as those that do it in the
conversion."""
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


def scenes():
    # violent coalescence: some ten bubbles are relabelled in every step
    return [S.random_bubbles(48, 48, 48, n_bubbles=80, r_min=2.0, r_max=5.0, u_max=0.2, sigma=1e-3, seed=seed) for seed in (0, 1)]


def run(fsl, precision, legs):
    """legs: (form, order, steps) one after the other."""
    sim = fsl.Simulation.from_scenarios(scenes(), precision=precision, split_trigger=1)
    relabelled = []
    for form, order, steps in legs:
        sim.set_interface_order(order)
        sim.set_stream_form(form)
        for _ in range(steps):
            sim.step(1)
            relabelled.append(sim.relabelled_bubbles)
    out = {"relabelled": relabelled}
    for d in range(2):
        for k, v in sim.fields(d, ("flags", "fill", "mass", "id", "pdf")).items():
            out[f"{k} {d}"] = v
        b = sim.bubbles(d)
        out[f"volume {d}"], out[f"pressure {d}"] = b["volume"], b["pressure"]
    sim.close()
    return out


def same(a, b, what):
    for k in a:
        assert np.array_equal(a[k], b[k]), f"{what}: {k}"


@pytest.mark.parametrize("form, order", [(5, 0), (5, 1), (8, 1)])
def test_fp64_state_is_that_of_the_split_form(fsl, form, order):
    same(run(fsl, "fp64", [(0, 0, 100)]), run(fsl, "fp64", [(form, order, 100)]), f"form {form}, order {order}")


@pytest.mark.parametrize("precision", ["fp32", "f16s", "bf16s"])
def test_two_kernel_forms_with_and_without_fused_fill_levels(fsl, precision):
    ref = run(fsl, precision, [(5, 0, 60)])
    for form in (5, 8):
        same(ref, run(fsl, precision, [(form, 1, 60)]), f"form {form} in order")


@pytest.mark.parametrize("form", [6, 7])
def test_tile_fused_step_relabels_the_same_bubbles(fsl, form):
    """One tile-fused step after k steps in form 5: a last bit cannot move a trigger."""
    for k in range(14, 34):
        a, b = run(fsl, "fp32", [(5, 0, k + 1)]), run(fsl, "fp32", [(5, 0, k), (form, 0, 1)])
        assert a["relabelled"] == b["relabelled"], f"after {k} steps"
        for d in range(2):
            assert np.array_equal(a[f"flags {d}"], b[f"flags {d}"]) and np.array_equal(a[f"id {d}"], b[f"id {d}"])
