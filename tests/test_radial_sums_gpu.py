"""The radial histogram behind the observables takes a point together with its
mirror images: states that live on single points (corners, axes, the rows and
columns without a mirror image, a generic point in each quadrant) must be
placed at their own radius, on grids smaller than a warp's share and stretched
ones.  With all atoms at one radius, R99 is the upper edge of its bin; a radius
within rounding (1e-9 bins) of an edge may fall on either side.  The separation
parameter is a ratio of FP64 sums of at most 8192 exactly widened values: 1e-12.
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


NPT = {"c64": np.complex64, "c128": np.complex128}
SIZES = [(8, 8, 4.0, 4.0), (8, 64, 2.0, 6.0), (256, 16, 20.0, 1.0), (64, 128, 8.0, 8.0)]


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("nx,ny,Lx,Ly", SIZES)
def test_single_points_are_placed_at_their_radius(dtype, nx, ny, Lx, Ly):
    g = inputs.Grid(nx, ny, Lx, Ly)
    X, Y = g.mesh()
    hx, hy = nx // 2, ny // 2
    pts = [(0, 0), (0, hx), (hy, 0), (hy, hx), (0, 1), (1, 0), (hy, 1), (hy - 1, hx), (1, 2), (1, nx - 2),
           (ny - 1, 2), (ny - 1, nx - 2), (hy - 1, hx + 1), (hy + 2, hx - 3), (hy, hx - 1), (hy + 1, 0)]
    psi = np.zeros((len(pts), 2, ny, nx), NPT[dtype])
    for k, (y, x) in enumerate(pts):
        psi[k, 0, y, x], psi[k, 1, y, x] = 1.5 - 0.5j, 0.25j
    with sp.Context(nx, ny, Lx, Ly, dtype, ninst=len(pts)) as c:
        got = c.observables(torch.from_numpy(psi).cuda())
    h = 0.5 * min(g.dx, g.dy)
    for k, (y, x) in enumerate(pts):
        r = np.hypot(X[y, x], Y[y, x]) / h
        assert got[k, 3] / h in [pytest.approx(np.floor(q) + 1, abs=1e-9) for q in (r - 1e-9, r + 1e-9)], (pts[k], r)
        assert abs(got[k, 0]) < 1e-12  # one point: the components overlap


@pytest.mark.parametrize("dtype", ["c64", "c128"])
@pytest.mark.parametrize("nx,ny,Lx,Ly", SIZES)
def test_sums_of_states_without_symmetry(orc, dtype, nx, ny, Lx, Ly):
    rng = np.random.default_rng(5)
    psi = (rng.normal(size=(3, 2, ny, nx)) + 1j * rng.normal(size=(3, 2, ny, nx))).astype(NPT[dtype])
    with sp.Context(nx, ny, Lx, Ly, dtype, ninst=3) as c:
        got = c.observables(torch.from_numpy(psi).cuda())
    m = orc.Model(nx, ny, Lx, Ly)
    g = inputs.Grid(nx, ny, Lx, Ly)
    for k in range(3):
        want = m.observables(psi[k].astype(np.complex128))
        assert abs(got[k, 0] - want[0]) < 1e-12
        assert abs(got[k, 3] - want[3]) <= 0.5 * min(g.dx, g.dy) + 1e-12
