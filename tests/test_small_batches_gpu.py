"""Batches with fewer row units or column tiles than the GPU has SMs: the passes
then run in smaller blocks.  Real-time steps must agree bit for bit with the
plain passes (SPGPE_PERSISTENT=0) at sizes around those rules' lines, ragged
ones among them, in both precisions; imaginary time, whose atom numbers are
added in another order, to rounding.
"""
import numpy as np
import pytest

import paper_2010_15069_gb300 as sp
from paper_2010_15069_gb300 import inputs

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA not available", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2010_15069_gb300 import build
    build.build()
    sp.load()


def run(monkeypatch, plain, dtype, nx, ny, ninst, imag):
    if plain:
        monkeypatch.setenv("SPGPE_PERSISTENT", "0")
    else:
        monkeypatch.delenv("SPGPE_PERSISTENT", raising=False)
    g = inputs.Grid(nx, ny, 8.0, 8.0)
    psi = np.stack([inputs.gaussian_spinor(g, width=1.5, noise=0.1, seed=i) for i in range(ninst)])
    t = torch.from_numpy(psi.astype(np.complex64 if dtype == "c64" else np.complex128)).cuda()
    p = inputs.problem(nx, ny, 8.0, 8.0, Omega=2.0, delta_slope=0.3, g11=100.0, g22=90.0, g12=95.0, kL=1.0)
    with sp.Context(nx, ny, 8.0, 8.0, dtype, ninst=ninst) as c:
        c.set_potentials_separable(**p.separable, g11=p.g11, g22=p.g22, g12=p.g12, kL=p.kL)
        if imag:
            c.step_imag(t, 1e-3, 6, lagged=True)
        else:
            c.step_real(t, 1e-3, 6)
        c.sync()
    return t.cpu().numpy()


# 64 x 64: one warp per block; 16 x 16 and 8 x 256: fewer units than SMs by far;
# 256 x 256 x 2: four warps per block; 32 x 512, 512 x 64: tall and wide tiles
@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("nx,ny,ninst", [(64, 64, 1), (16, 16, 1), (8, 256, 1), (256, 256, 2), (32, 512, 3), (512, 64, 1),
                                         (128, 128, 9)])
def test_small_batches_agree_with_the_plain_passes(monkeypatch, dtype, nx, ny, ninst):
    a, b = (run(monkeypatch, plain, dtype, nx, ny, ninst, False) for plain in (False, True))
    assert np.array_equal(a, b)
    a, b = (run(monkeypatch, plain, dtype, nx, ny, ninst, True) for plain in (False, True))
    assert np.abs(a - b).max() < (2e-6 if dtype == "c64" else 1e-14)
