"""Two and four kept modes, the fewest that the truncated transforms' own kernels
take: a block of the transform along y then holds many images, and its shared
memory has to bound their number.  Forward pass, every gradient and an Adam
step against the FP64 oracle, with the tolerances of the network's other parity
tests (float32 accumulation error).
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


# (width, modes, hidden, n, batch): batches that leave a block's images short among them
@pytest.mark.parametrize("W,M,H,n,B", [(32, 2, 64, 64, 1), (32, 2, 64, 64, 9), (64, 2, 128, 128, 2), (32, 4, 48, 64, 3)])
def test_few_modes_match_the_oracle(W, M, H, n, B):
    rng = np.random.default_rng(W + M + n + B)
    sh = ofno.Shapes(3, 4, W, M, 2, H)
    a = rng.standard_normal((B, 3, n, n)).astype(np.float32)
    t = rng.standard_normal((B, 4, n, n)).astype(np.float32)
    with sp.FNO(3, 4, width=W, modes=M, layers=2, hidden=H, seed=3) as f:
        theta = (f.get_params() + rng.uniform(-0.05, 0.05, f.num_params())).astype(np.float32)
        f.set_params(theta)
        ad, td = torch.from_numpy(a).cuda(), torch.from_numpy(t).cuda()
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
