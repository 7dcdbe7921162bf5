"""The allocation-free labelling at its size limit of 2^21 cells, on the lattices
with the most unions that meet: full, checkerboard (connected over edges only), and
a random one near the percolation threshold."""
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


@pytest.mark.parametrize("dims", [(128, 128, 128), (4096, 32, 16), (2, 1024, 1024)])
@pytest.mark.parametrize("kind", ["full", "checkerboard", "random"])
def test_labels_at_the_size_limit(fsl, oracle_mod, dims, kind):
    import torch
    nx, ny, nz = dims
    z, y, x = np.ogrid[:nz, :ny, :nx]
    if kind == "full":
        fg = np.ones((nz, ny, nx), dtype=bool)
    elif kind == "checkerboard":
        fg = np.broadcast_to((x + y + z) % 2 == 0, (nz, ny, nx)).copy()
    else:
        fg = np.random.Generator(np.random.PCG64(4)).uniform(size=(nz, ny, nx)) < 0.14
    want = np.asarray(oracle_mod.label(fg)).reshape(-1)
    flags = torch.from_numpy(np.where(fg, S.GAS, S.LIQUID).astype(np.uint8).reshape(-1)).cuda()
    out = torch.empty(nx * ny * nz, dtype=torch.int64, device="cuda")
    for _ in range(5):
        out.fill_(-7)
        fsl.label_bubbles_static(flags, nx, ny, nz, out)
        assert np.array_equal(out.cpu().numpy(), want)
