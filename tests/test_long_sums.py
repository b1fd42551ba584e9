"""Per-thread FP32 sums of the register x passes (reduce.cuh), compiled for the host.

A thread of the inverse pass may hold 200 elements of an inner product.  Its total, from
chunks of 8, has to stay within 8 x 2^-24 of the sum of the magnitudes however many there
are: 7 additions within a chunk and the last one.  (With each product's own rounding and
the tree over the block that is the 16 x 2^-24 of a kernel with 8 elements a thread.)
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1305_6497_gb300", "csrc")
PROGRAM = """
#include <cstdio>
#include "reduce.cuh"
int main() {
  int n;
  while (scanf("%d", &n) == 1) {
    dda::LongAcc<2> acc;
    for (int i = 0; i < n; ++i) {
      float v;
      if (scanf("%f", &v) != 1) return 1;
      acc.add(0, v);
      acc.add(1, -v);
      if (i % 8 == 7) acc.flush();
    }
    acc.flush();
    printf("%.9g %.9g\\n", acc.total(0), acc.total(1));
  }
}
"""


@pytest.fixture(scope="module")
def total(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    d = tmp_path_factory.mktemp("sums")
    (d / "sums.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-arch=sm_103a", "-I", CSRC,
                    "-o", str(d / "sums"), str(d / "sums.cu")], check=True, capture_output=True)

    def run(values):
        text = f"{len(values)} " + " ".join(f"{v:.9g}" for v in values)
        out = subprocess.run([str(d / "sums")], input=text, capture_output=True, text=True,
                             check=True).stdout.split()
        assert float(out[0]) == -float(out[1])
        return float(out[0])
    return run


@pytest.mark.parametrize("n", [1, 8, 9, 16, 128, 250, 4000])
@pytest.mark.parametrize("kind", ["random", "positive", "lost", "cancelling"])
def test_error_does_not_grow_with_the_number_of_elements(total, n, kind):
    rng = np.random.default_rng(n)
    v = rng.standard_normal(n).astype(np.float32)
    if kind == "positive":
        v = np.abs(v)
    elif kind == "lost":            # every chunk after the first below half an ulp of the total
        v[:] = 0
        v[::8] = 0.98 * 2.0 ** -24
        v[0] = 1
    elif kind == "cancelling":
        v[n // 2:] = -v[:n - n // 2]
    exact = np.sum(v.astype(np.float64))
    assert abs(total(v) - exact) <= 8 * 2.0 ** -24 * np.sum(np.abs(v.astype(np.float64)))
