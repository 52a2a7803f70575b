"""The double-precision series of the pointwise operators over their own ranges
(csrc/fastmath.cuh: expm1 below 1/32 and 1/4, the shear constants tan h and sin 2h
below 1/64 and 1/8), against extended precision.  Inside the range: 3 x 2^-52
relative (the series' first omitted term is below 1e-17, the rest is the rounding
of a Horner chain whose last steps dominate).  Beyond it, up to 1: within 1.5 times
the first omitted term, which an error in any coefficient, also the highest,
would exceed.
"""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():  # pragma: no cover
    pytest.skip("CUDA not available", allow_module_level=True)

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
SRC = os.path.join(HERE, "csrc", "fastmath64_probe.cu")
CSRC = os.path.join(ROOT, "paper_2010_15069_gb300", "csrc")
LIB = os.path.join(HERE, "_build", "libfastmath64_probe.so")


@pytest.fixture(scope="module")
def probe():
    from paper_2010_15069_gb300 import build
    os.makedirs(os.path.dirname(LIB), exist_ok=True)
    tmp = LIB + f".tmp{os.getpid()}"
    subprocess.run([build.nvcc(), "-std=c++17", "-O3", *build.ARCH, "-Xcompiler", "-fPIC", "-shared", "-I", CSRC, SRC,
                    "-o", tmp], check=True)
    os.replace(tmp, LIB)
    lib = ctypes.CDLL(LIB)
    lib.fastmath64_probe.argtypes = [ctypes.c_int, ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]

    def run(fn, x):
        xd = torch.from_numpy(np.ascontiguousarray(x, dtype=np.float64)).cuda()
        out = torch.zeros(2 * x.size, dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert lib.fastmath64_probe(fn, xd.data_ptr(), x.size, out.data_ptr()) == 0
        return out.cpu().numpy().reshape(-1, 2)
    return run


def tan_coefficient(k):
    """Coefficient of h^(2k - 1) in tan h, by its derivatives' recurrence y' = 1 + y^2."""
    from fractions import Fraction
    c = [Fraction(0)] * (2 * k)
    c[1] = Fraction(1)
    for n in range(2, 2 * k):
        s = sum(c[i] * c[n - 1 - i] for i in range(n))
        c[n] = s / n
    return float(c[2 * k - 1])


# (function, output, exact, limit, first omitted term relative to the leading one)
CASES = [
    (0, 0, np.expm1, 1 / 32, lambda x: x ** 9 / math.factorial(10)),
    (1, 0, np.expm1, 1 / 4, lambda x: x ** 13 / math.factorial(14)),
    (2, 0, np.tan, 1 / 64, lambda x: x ** 10 * tan_coefficient(6)),
    (2, 1, lambda h: np.sin(2 * h), 1 / 64, lambda x: (2 * x) ** 8 / math.factorial(9)),
    (3, 0, np.tan, 1 / 8, lambda x: x ** 16 * tan_coefficient(9)),
    (3, 1, lambda h: np.sin(2 * h), 1 / 8, lambda x: (2 * x) ** 12 / math.factorial(13)),
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_series_over_their_ranges(probe, case):
    fn, col, exact, limit, omitted = CASES[case]
    a = np.concatenate([np.linspace(limit * 1e-4, limit, 100001), np.logspace(-300, np.log10(limit), 4001),
                        np.linspace(limit, 1.0, 2001)])
    x = np.concatenate([a, -a])
    got = probe(fn, x)[:, col].astype(np.longdouble)
    ref = exact(x.astype(np.longdouble))
    lead = np.abs(x) * (2 if col == 1 else 1)
    err = (np.abs(got - ref) / lead).astype(np.float64)
    inside = np.abs(x) <= limit
    bound = 3 * 2.0 ** -52 + 1.5 * omitted(np.abs(x)) * np.where(inside, 1.0, grow(case, np.abs(x)))
    assert np.all(err <= bound), (x[np.argmax(err / bound)], np.max(err / bound))
    assert omitted(limit) < 1e-17


def grow(case, x):
    """The tail's sum over its first term: geometric with the ratio of the next terms at |x| <= 1."""
    if CASES[case][2] is np.tan:
        return 1 / (1 - (x / (math.pi / 2)) ** 2)  # tan's coefficients fall by (2 / pi)^2
    return 1.0
