"""complex128 batches whose column passes run in narrowed tiles (fewer blocks than
the GPU has SMs): against the FP64 oracle, in real and imaginary time, and an
instance alone against the same one inside a batch whose tiles are not narrowed,
bit for bit.
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


SIZES = [(16, 16), (64, 64), (8, 256), (512, 64), (32, 512), (128, 128), (16, 2048)]


def problem(nx, ny):
    return inputs.problem(nx, ny, 8.0, 8.0, Omega=2.0, delta_slope=0.3, g11=100.0, g22=90.0, g12=95.0, kL=1.0)


def run(p, psi, imag, steps=4, dt=1e-3):
    g = p.grid
    with sp.Context(g.nx, g.ny, 8.0, 8.0, "c128", ninst=len(psi)) as c:
        c.set_potentials_separable(**p.separable, g11=p.g11, g22=p.g22, g12=p.g12, kL=p.kL)
        t = torch.from_numpy(psi).cuda()
        (c.step_imag if imag else c.step_real)(t, dt, steps)
        c.sync()
    return t.cpu().numpy()


@pytest.mark.parametrize("imag", [False, True])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_narrowed_tiles_match_the_oracle(orc, nx, ny, imag):
    p = problem(nx, ny)
    psi = np.stack([inputs.gaussian_spinor(p.grid, width=1.5, noise=0.1, seed=i) for i in range(2)])
    got = run(p, psi, imag)
    m = orc.Model(nx, ny, 8.0, 8.0, V=p.V, delta=p.delta, Omega=p.Omega, g11=p.g11, g22=p.g22, g12=p.g12, kL=p.kL)
    for k in range(2):
        ref = m.step(psi[k], 1e-3, 4, imag=imag, norm_mode=0, target=(0.5, 0.5))
        assert np.abs(got[k] - ref).max() < 1e-13


@pytest.mark.parametrize("nx,ny", SIZES)
def test_an_instance_alone_and_in_a_large_batch(nx, ny):
    p = problem(nx, ny)
    one = inputs.gaussian_spinor(p.grid, width=1.5, noise=0.1, seed=7)[None]
    tiles = max(1, nx // 8) * 2
    many = np.repeat(one, -(-304 // tiles), axis=0)
    assert np.array_equal(run(p, one, False)[0], run(p, many, False)[-1])
