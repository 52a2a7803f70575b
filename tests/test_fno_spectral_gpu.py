"""The spectral layers' own kernels against the FP64 oracle (oracle/fno.py) at the
sizes where their tiling can go wrong: both channel widths they cover, mode
counts that leave padded rows or are odd, batches around the samples that a
block holds, and the smallest grid and larger ones; and the Adam step of the
spectral weights, which is taken without a gradient in memory.
"""
import numpy as np
import pytest

import paper_2010_15069_gb300 as sp
from oracle import fno as ofno

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA not available", allow_module_level=True)


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2010_15069_gb300 import build
    build.build()
    sp.load()


def rel(x, y):
    return float(np.linalg.norm(np.ravel(x - y)) / max(np.linalg.norm(np.ravel(y)), 1e-30))


# (width, modes, layers, hidden, n, batch)
SHAPES = [(32, 12, 2, 64, 64, 9), (32, 6, 2, 64, 64, 1), (64, 10, 1, 128, 64, 3), (32, 16, 1, 64, 128, 5),
          (32, 5, 1, 64, 64, 2), (64, 24, 1, 128, 256, 1), (64, 32, 1, 128, 64, 2), (64, 32, 2, 128, 256, 4),
          (32, 16, 2, 48, 128, 2)]


def test_rows_of_several_segments():
    """512-point rows take two segments of the transform tables, and every block
    walks several tiles of each; inference against the oracle."""
    W, M, n, B = 64, 32, 512, 2
    rng = np.random.default_rng(8)
    sh = ofno.Shapes(3, 4, W, M, 1, 128)
    a = rng.standard_normal((B, 3, n, n)).astype(np.float32)
    with sp.FNO(3, 4, width=W, modes=M, layers=1, hidden=128, seed=3) as f:
        w = ofno.round_bf16(f.get_params().astype(np.float64))
        out = f.forward(torch.from_numpy(a).cuda()).cpu().numpy()
    assert rel(out, ofno.forward(sh, w, a.astype(np.float64))) < 2e-5


@pytest.mark.parametrize("W,M,L,H,n,B", SHAPES)
def test_gradients_and_optimiser_step(W, M, L, H, n, B):
    """Forward pass, loss, every gradient (float32 accumulation error: the
    tolerances of the network's other parity tests) and the weights after one
    Adam step against the update rule applied to the library's gradient."""
    rng = np.random.default_rng(W + M + n + B)
    sh = ofno.Shapes(3, 4, W, M, L, H)
    a = rng.standard_normal((B, 3, n, n)).astype(np.float32)
    t = rng.standard_normal((B, 4, n, n)).astype(np.float32)
    with sp.FNO(3, 4, width=W, modes=M, layers=L, hidden=H, seed=3) as f:
        theta = f.get_params().astype(np.float64)
        theta = (theta + rng.uniform(-0.05, 0.05, theta.size)).astype(np.float32)
        f.set_params(theta)
        ad, td = torch.from_numpy(a).cuda(), torch.from_numpy(t).cuda()
        out = f.forward(ad).cpu().numpy()
        loss, g, out2 = f.gradient(ad, td)
        f.train_step(ad, td, 1e-3)
        new = f.get_params().astype(np.float64)
    assert np.array_equal(out, out2.cpu().numpy())
    w = ofno.round_bf16(theta.astype(np.float64))
    assert rel(out, ofno.forward(sh, w, a.astype(np.float64))) < 2e-5
    lo, go = ofno.loss_and_grad(sh, w, a.astype(np.float64), t.astype(np.float64))
    assert abs(loss - lo) < 1e-5 * lo
    gd, god = sh.unpack(g), sh.unpack(go)
    for name, _ in sh.layout():
        assert rel(gd[name], god[name]) < 2e-4, name
    th = theta.astype(np.float64)
    want, _, _ = ofno.adam_step(th, g.astype(np.float64), np.zeros_like(th), np.zeros_like(th), 1, 1e-3)
    assert np.abs(new - want).max() < 1e-6
