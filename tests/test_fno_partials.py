"""The workspace of the network's gradient partials, on the CPU.

Every block of a weight-gradient product leaves its partial sums of the weight
and of the bias in one workspace, sized when a batch and a grid size are first
met.  A small host program compiled against the header (fno_internal.h)
evaluates the size and the demand of each product for networks whose output,
hidden and channel counts are larger and smaller than one another; the demand
has to fit, also for every smaller batch, which reuses the workspace.
"""
import itertools
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2010_15069_gb300", "csrc")

CHECK = r"""
#include <cstdio>
#include "fno_internal.h"
using namespace spgpe::fno;
int main() {
  int cin, cout, w, h, batch, n, sms;
  while (scanf("%d %d %d %d %d %d %d", &cin, &cout, &w, &h, &batch, &n, &sms) == 7) {
    const long P = (long)n * n;
    printf("%zu %d %d\n", partial_floats(cin, cout, w, h, batch, P, sms), weight_grad_parts(batch, P, sms),
           project_parts(batch, P, sms));
  }
  return 0;
}
"""


def _nvcc():
    for c in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and os.path.exists(c):
            return c
    return None


def test_every_product_fits_the_workspace(tmp_path):
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "check.cu", tmp_path / "check"
    src.write_text(CHECK)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src), "-o",
                    str(exe)], check=True, timeout=900)
    nets = [(3, 64, 32, 32), (6, 100, 64, 64), (3, 4, 2, 2), (3, 32, 8, 16), (6, 4, 64, 128), (200, 1, 8, 8), (1, 1024, 1, 1),
            (3, 4, 32, 64), (3, 128, 128, 128), (1, 1, 1, 128)]
    cases = [net + (b, n, sms) for net, b, n, sms in itertools.product(nets, (1, 3, 4, 8), (8, 64, 128, 256, 1024), (148, 152))]
    r = subprocess.run([str(exe)], input="\n".join(" ".join(map(str, c)) for c in cases), capture_output=True, text=True,
                       timeout=60, check=True)
    held = {}
    for c, line in zip(cases, r.stdout.splitlines(), strict=True):
        cin, cout, w, h, b, n, sms = c
        held[c], parts, heads = map(int, line.split())
        need = [heads * (cout * h + h + cout)]
        for m, k in ((w, cin), (w, w), (h, w), (cout, h)):
            need += [parts * (m * k + m), b * max(1, n * n // 1024) * m * k]
        assert held[c] >= max(need), c
    for c in cases:  # a smaller batch on the same grid
        if c[4] > 1:
            assert held[c[:4] + (1,) + c[5:]] <= held[c], c
