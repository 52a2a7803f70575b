"""Gradients of networks with more outputs than hidden units and channels, at
batches that give every block of the weight-gradient products work: the
partial sums of the output layer (a weight and a bias per block) are the
largest of the network, and have to fit their workspace.  Against the FP64
oracle, with the tolerances of the network's other parity tests.
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


@pytest.mark.parametrize("cin,cout,W,M,H,n,B", [(3, 64, 32, 4, 32, 128, 8), (6, 100, 64, 4, 64, 128, 4),
                                                (3, 4, 2, 3, 2, 64, 8), (3, 32, 8, 4, 16, 64, 5)])
def test_gradients_with_many_outputs(cin, cout, W, M, H, n, B):
    rng = np.random.default_rng(cout + n)
    sh = ofno.Shapes(cin, cout, W, M, 1, H)
    a = rng.standard_normal((B, cin, n, n)).astype(np.float32)
    t = rng.standard_normal((B, cout, n, n)).astype(np.float32)
    with sp.FNO(cin, cout, width=W, modes=M, layers=1, hidden=H, seed=3) as f:
        theta = (f.get_params() + rng.uniform(-0.05, 0.05, f.num_params())).astype(np.float32)
        f.set_params(theta)
        loss, g, _ = f.gradient(torch.from_numpy(a).cuda(), torch.from_numpy(t).cuda())
    lo, go = ofno.loss_and_grad(sh, ofno.round_bf16(theta.astype(np.float64)), a.astype(np.float64), t.astype(np.float64))
    assert abs(loss - lo) < 1e-5 * lo
    gd, god = sh.unpack(g), sh.unpack(go)
    for name, _ in sh.layout():
        assert rel(gd[name], god[name]) < 2e-4, name
