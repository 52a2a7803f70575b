"""Imaginary-time steps whose Raman rotation makes the density grow between the
point where a pass bounds the interaction exponent and the factors that use
it: the series that the bound picks must still hold.
An antisymmetric spinor (the growing eigenvector of exp(-theta sigma_x)) whose
exponent before the rotation lies just below each tier's bound, against the FP64
oracle within the rounding of a step: complex128 1e-13 (entries below 1),
complex64 the tolerance of its other step tests, 2e-6.  One step: where the peak is
saturated and the tails grow by exp(5) a step, later steps amplify the transforms'
rounding noise in the tails (twelvefold a step, the same in both precisions).
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


# target: the interaction exponent before the rotation, dt / 2 * 1.9 g * 1.05 * (2 / pi at the peak), just below
# 1/32, 1/4 and 1/2; omega dt = 10 multiplies the densities by exp(2.5) in the opening rotation alone
@pytest.mark.parametrize("dtype", ["c128", "c64"])
@pytest.mark.parametrize("two_d", [False, True])
@pytest.mark.parametrize("target", [0.03, 0.24, 0.48])
@pytest.mark.parametrize("omega,V0", [(1000.0, 0.0), (300.0, -200.0), (5.0, 0.0)])
def test_growing_densities_match_the_oracle(orc, dtype, two_d, target, omega, V0):
    n, box, dt, steps = 64, 8.0, 1e-2, 1
    g = target / (0.5 * dt * 1.9 * 1.05 * 2 / np.pi)
    p = inputs.problem(n, n, box, box, Omega=omega, delta_slope=0.1, g11=g, g22=g, g12=0.9 * g, kL=0.5)
    u = inputs.gaussian_spinor(p.grid, width=1 / np.sqrt(2.0), noise=1e-2, seed=4)[0]
    psi0 = np.stack([u, -u])
    V = p.V + V0
    with sp.Context(n, n, box, box, dtype) as c:
        if two_d:
            c.set_potentials(V, p.delta, p.Omega, p.g11, p.g22, p.g12, p.kL)
        else:
            s = dict(p.separable)
            s["Vy"] = s["Vy"] + V0
            c.set_potentials_separable(**s, g11=p.g11, g22=p.g22, g12=p.g12, kL=p.kL)
        t = torch.from_numpy(psi0.astype(np.complex64 if dtype == "c64" else np.complex128)).cuda()
        c.step_imag(t, dt, steps)
        c.sync()
    m = orc.Model(n, n, box, box, V=V, delta=p.delta, Omega=p.Omega, g11=p.g11, g22=p.g22, g12=p.g12, kL=p.kL)
    ref = m.step(psi0, dt, steps, imag=True, norm_mode=0, target=(0.5, 0.5))
    assert np.abs(t.cpu().numpy() - ref).max() < (1e-13 if dtype == "c128" else 2e-6)
