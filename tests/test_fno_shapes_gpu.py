"""Network shapes that mix the fused kernels with the general products: widths
beside 32 and 64, hidden widths beside twice the width, one output and more than
four, many inputs, and an input at an address that is not 16-byte aligned.
Forward pass, gradients and an Adam step against the FP64 oracle, with the
tolerances of the network's other parity tests.
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


def device(x, offset):
    """x on the GPU, `offset` floats past an aligned address."""
    buf = torch.empty(x.size + offset, dtype=torch.float32, device="cuda")
    t = buf[offset:].view(x.shape)
    t.copy_(torch.from_numpy(x))
    return t


# (cin, cout, width, modes, hidden, n, batch, offset)
@pytest.mark.parametrize("cin,cout,W,M,H,n,B,offset", [
    (3, 4, 96, 4, 192, 64, 2, 0), (3, 4, 128, 6, 128, 64, 2, 0), (9, 1, 16, 4, 32, 64, 3, 0), (9, 5, 32, 8, 64, 64, 2, 0),
    (3, 1, 64, 8, 128, 64, 2, 0), (3, 4, 64, 8, 64, 64, 2, 0), (3, 4, 32, 8, 128, 64, 2, 0), (3, 4, 32, 8, 64, 64, 2, 1),
    (3, 4, 64, 6, 128, 128, 1, 3)])
def test_mixed_shapes_match_the_oracle(cin, cout, W, M, H, n, B, offset):
    rng = np.random.default_rng(W + H + cin)
    sh = ofno.Shapes(cin, cout, W, M, 2, H)
    a = rng.standard_normal((B, cin, n, n)).astype(np.float32)
    t = rng.standard_normal((B, cout, n, n)).astype(np.float32)
    with sp.FNO(cin, cout, width=W, modes=M, layers=2, hidden=H, seed=3) as f:
        theta = (f.get_params() + rng.uniform(-0.05, 0.05, f.num_params())).astype(np.float32)
        f.set_params(theta)
        ad, td = device(a, offset), device(t, offset)
        out = f.forward(ad).cpu().numpy()
        loss, g, _ = f.gradient(ad, td)
        f.train_step(ad, td, 1e-3)
        new = f.get_params().astype(np.float64)
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
