"""The allocation-free labelling on ragged lattices against the oracle's flood
fill."""
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


@pytest.mark.parametrize("dims", [(1, 1, 7), (2, 3, 5), (31, 9, 4), (32, 8, 8), (33, 5, 6), (64, 3, 3), (95, 17, 13),
                                  (256, 4, 2)])
@pytest.mark.parametrize("share", [0.08, 0.4, 0.97, 1.0])
def test_static_labels_of_ragged_lattices(fsl, oracle_mod, dims, share):
    """Rows shorter and longer than a warp, rows that straddle warps, rows full of
    bubble cells (a run that closes on itself through the wrap), single cells."""
    import torch
    nx, ny, nz = dims
    rng = np.random.Generator(np.random.PCG64(nx * 1000 + ny))
    fg = rng.uniform(size=(nz, ny, nx)) < share
    flags = np.where(fg, np.where(rng.uniform(size=fg.shape) < 0.5, S.GAS, S.INTERFACE), S.LIQUID).astype(np.uint8)
    want = oracle_mod.label(fg)
    dev = torch.from_numpy(flags.reshape(-1)).cuda()
    out = torch.full((nx * ny * nz,), -7, dtype=torch.int64, device="cuda")
    fsl.label_bubbles_static(dev, nx, ny, nz, out)
    assert np.array_equal(out.cpu().numpy(), np.asarray(want).reshape(-1))
