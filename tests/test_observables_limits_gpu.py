"""The radial histogram at the sizes where its shared memory meets a limit: around
48 KB, up to which a block needs no grant, and near the largest that a block may
have.  States on single points lie in the bin of their own radius (R99 is its
upper edge).
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


# bins: the box's corner radius over half a grid step, plus two
@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("Lx,nb", [(0.3, 68), (93.975, 6016), (93.98, 6017), (94.5, 6050), (95.96, 6143), (96.0, 6146), (452.0, 28930),
                                   (453.1, 29000)])
def test_histograms_around_the_shared_memory_limits(dtype, Lx, nb):
    nx, ny, Ly = 8, 64, 1.0
    g = inputs.Grid(nx, ny, Lx, Ly)
    h = 0.5 * min(g.dx, g.dy)
    if nb > 68:
        assert int(np.hypot(Lx, Ly) / h) + 2 == nb
    X, Y = g.mesh()
    pts = [(0, 0), (0, 4), (32, 1), (33, 2), (31, 7), (60, 5), (5, 3)]
    psi = np.zeros((len(pts), 2, ny, nx), np.complex64 if dtype == "c64" else np.complex128)
    for k, (y, x) in enumerate(pts):
        psi[k, 0, y, x], psi[k, 1, y, x] = 1.5 - 0.5j, 0.25j
    with sp.Context(nx, ny, Lx, Ly, dtype, ninst=len(pts)) as c:
        got = c.observables(torch.from_numpy(psi).cuda())
    for k, (y, x) in enumerate(pts):
        r = np.hypot(X[y, x], Y[y, x]) / h
        assert got[k, 3] / h in [pytest.approx(np.floor(q) + 1, abs=1e-6) for q in (r - 1e-9, r + 1e-9)], (pts[k], r)
