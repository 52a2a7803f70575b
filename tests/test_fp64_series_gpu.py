"""The double-precision series of the pointwise operators: complex128 steps whose
phases or exponents fall into each tier (below 1/64, below 1/8 and beyond in
real time; below 1/32, below 1/4 and beyond in imaginary time) against the FP64
oracle, within the rounding of a few steps.
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


# peak density 1 / pi per component of half an atom and width 1 / sqrt 2: the
# interaction exponent dt / 2 (g11 + g12) / pi is 0.013, 0.13 and 1.3 for the three
# couplings in imaginary time; in real time the largest half phase is about the
# trap's, dt / 4 * 32 = 0.008, 0.08, 0.8 for the three steps
@pytest.mark.parametrize("imag,dt,g", [(True, 2e-3, 20.0), (True, 2e-3, 200.0), (True, 2e-3, 2000.0),
                                       (False, 1e-3, 2.0), (False, 1e-2, 2.0), (False, 1e-1, 2.0)])
def test_double_precision_tiers_match_the_oracle(orc, imag, dt, g):
    n, box, steps = 64, 8.0, 5
    p = inputs.problem(n, n, box, box, Omega=0.5, delta_slope=0.1, g11=g, g22=g, g12=0.9 * g, kL=0.5)
    psi0 = inputs.gaussian_spinor(p.grid, width=1 / np.sqrt(2.0), noise=1e-2, seed=4)
    with sp.Context(n, n, box, box, "c128") as c:
        c.set_potentials_separable(**p.separable, g11=p.g11, g22=p.g22, g12=p.g12, kL=p.kL)
        t = torch.from_numpy(psi0.copy()).cuda()
        (c.step_imag if imag else c.step_real)(t, dt, steps)
        c.sync()
    g0 = p.grid
    m = orc.Model(g0.nx, g0.ny, g0.xmax, g0.ymax, V=p.V, delta=p.delta, Omega=p.Omega, g11=p.g11, g22=p.g22, g12=p.g12,
                  kL=p.kL)
    ref = m.step(psi0, dt, steps, imag=imag, norm_mode=0, target=(0.5, 0.5))
    assert np.abs(t.cpu().numpy() - ref).max() < 1e-13
