"""FP32 and 16-bit storage: the stream-collide forms of one family (0-4, 5 and 8, 6
and 7) give one state, bit for bit, and the tuner takes a form of the family that
the size of the workload names, whatever ran before in the process."""
import numpy as np
import pytest

from paper_1604_01632_gb300 import scenarios as S

pytestmark = pytest.mark.gpu
FAMILIES = [(0, 1, 2, 3, 4), (5, 8), (6, 7)]


@pytest.fixture(scope="module")
def fsl():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1604_01632_gb300 import build, fsl as F
    build.build()
    return F


def bubbles(dims, seed, per_cell=4e-4, u_max=0.1):
    n = dims[0] * dims[1] * dims[2]
    return S.random_bubbles(*dims, n_bubbles=max(2, int(per_cell * n)), r_min=3.0, r_max=7.0, u_max=u_max, sigma=4e-3,
                            seed=seed)


SHAPES = {"one": [(64, 60, 56)], "odd rows": [(61, 47, 53)], "batch": [(33, 40, 29), (32, 48, 40)]}


@pytest.mark.parametrize("order", [0, 1])
@pytest.mark.parametrize("precision", ["fp32", "f16s", "bf16s"])
@pytest.mark.parametrize("shape", list(SHAPES))
def test_one_state_per_family(fsl, shape, precision, order):
    scs = [bubbles(dims, d) for d, dims in enumerate(SHAPES[shape])]
    for family in FAMILIES:
        ref = None
        for form in family:
            if form == 4 and not order:
                continue
            sim = fsl.Simulation.from_scenarios(scs, precision=precision)
            sim.set_interface_order(order)
            sim.set_stream_form(form)
            sim.step(30)
            got = [sim.fields(d, ("flags", "fill", "mass", "id", "pdf")) for d in range(len(scs))]
            sim.close()
            if ref is None:
                ref = got
                continue
            for d, (x, y) in enumerate(zip(ref, got)):
                for name in x:
                    assert np.array_equal(x[name], y[name]), f"forms {family[0]} and {form}, domain {d}, {name}"


def tuned(fsl, scs, precision):
    sim = fsl.Simulation.from_scenarios(scs, precision=precision)
    sim.step(20)
    form = sim.tuning()["form"]
    sim.close()
    return form


# lattices whose family has not always been the fastest one, some 10 % interface cells
@pytest.mark.parametrize("dims, precision, family", [
    ((61, 47, 53), "fp32", 0), ((58, 56, 56), "f16s", 0), ((62, 60, 58), "bf16s", 2), ((80, 80, 80), "f16s", 2), ((88, 88, 88), "bf16s", 2),
    ((96, 96, 96), "fp32", 2)])
def test_the_tuner_keeps_to_the_family(fsl, dims, precision, family):
    scs = [bubbles(dims, 1, u_max=0.03)]
    L = fsl.load_library()
    for _ in range(3):
        L.fsl_forget_tuning()
        assert tuned(fsl, scs, precision) in FAMILIES[family]


def test_a_cached_form_is_of_the_same_family(fsl):
    """Two lattices of one cache key (FP32, 2^22 to 2^23 cells, 6/64 interface), either
    one first."""
    foams = {n: [S.foam(n, seed=2)] for n in (164, 192)}      # 4.4 M and 7.1 M cells
    for sides in ((192, 164), (164, 192)):
        fsl.load_library().fsl_forget_tuning()
        for n in sides:
            assert tuned(fsl, foams[n], "fp32") in FAMILIES[2]
