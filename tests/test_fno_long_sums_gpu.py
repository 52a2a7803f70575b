"""Weight and bias gradients over 8.4 million points, where the length of a running
sum shows: with constant fields every term of a gradient is the same number, so
rounding errors of one sign add up instead of averaging out.

The network has constant activations (no input map, no spectral weights, large
hidden biases, for which the GELU is the identity), so that every gradient is
the number of points times a product of known values; the target holds small
integers, whose squares sum exactly.  Bounds, relative, from the longest chain a
partial sum may have, 16 blocks of 64 points: operands kept to 16 bits (2^-16) and
64 accumulation steps of two products that each truncate (128 x 2^-23): 3.1e-5.
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


# the general products, and the fused lift, layer and projection: (width, modes, hidden, outputs)
NETS = [(8, 1, 16, 8), (32, 4, 64, 4)]


def relative_errors(W, M, H, C):
    """Largest relative error of each gradient tensor of a network of constant fields."""
    n, B = 1024, 8
    rng = np.random.default_rng(W)

    def bf(*shape):  # positive values with the 8 bits of a bfloat16
        return ofno.round_bf16(rng.uniform(0.5, 1.0, shape))

    sh = ofno.Shapes(1, C, W, M, 1, H)
    p = {name: np.zeros(shape) for name, shape in sh.layout()}
    p["p"], p["w0"], p["Q1"], p["q1"] = bf(W), bf(W), bf(H, W) / 16, 32 + 16 * bf(H)
    p["q1"], p["Q2"], p["q2"] = ofno.round_bf16(p["q1"]), bf(C, H) / 1024, ofno.round_bf16(-20 - 4 * bf(C))
    t = np.arange(C) % 3 + 1.0
    with sp.FNO(1, C, width=W, modes=M, layers=1, hidden=H, seed=3) as f:
        f.set_params(sh.pack(p).astype(np.float32))
        ad = torch.zeros(B, 1, n, n, device="cuda")
        td = torch.from_numpy(t.astype(np.float32)).cuda().view(1, C, 1, 1).expand(B, C, n, n).contiguous()
        _, g, out = f.gradient(ad, td)
        o = out[:, :, :1, :1].clone()
        assert bool((out == o).all())  # constant fields indeed
        o = o[0, :, 0, 0].cpu().numpy().astype(np.float64)
    d = ((o - t) * (2.0 / (n * n * np.sum(t * t)) / B)).astype(np.float32).astype(np.float64)
    h = p["Q1"] @ p["w0"] + p["q1"]
    dh = p["Q2"].T @ d
    dv = p["Q1"].T @ dh
    want = {"q2": d, "Q2": np.outer(d, h), "q1": dh, "Q1": np.outer(dh, p["w0"]), "w0": dv, "W0": np.outer(dv, p["p"])}
    got = sh.unpack(g)
    return {k: float(np.abs(got[k] / (B * n * n * want[k]) - 1.0).max()) for k in want}


@pytest.mark.parametrize("net", NETS)
def test_weight_gradients_of_constant_fields(net):
    err = relative_errors(*net)
    assert all(err[k] < 3.1e-5 for k in ("Q2", "Q1", "W0")), err


@pytest.mark.parametrize("net", NETS)
def test_bias_gradients_of_constant_fields(net):
    """16 additions of sums over 8 points (3) and 8 or 32 lanes (3 to 5), and up to 8
    terms of the hidden gradient behind each value: 32 x 2^-24 = 2e-6; dw0 in addition
    the 24 tensor-core steps of the transposed map: + 24 x 2^-23; the fused
    projection's dQ2, 64 + 5 + 8 float32 steps: 4.6e-6."""
    err = relative_errors(*net)
    assert err["q2"] < 2e-6 and err["q1"] < 2e-6 and err["w0"] < 5e-6, err
    if net[2] == 2 * net[0] and net[0] >= 32:
        assert err["Q2"] < 4.6e-6, err
