"""The compensated sums of the adjoint's scalars (csrc/dg_sum2.h), compiled for the CPU: sums by quarters of terms that
cancel against the exact sum."""
import math
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HARNESS = r"""
#include <cstdio>
#include <vector>
#include "dg_sum2.h"
// stdin: runs of n, stride, factor, n x stride floats; stdout: the joined quarters, and the same scaled
int main() {
  int n, st;
  float k;
  while (std::scanf("%d %d %f", &n, &st, &k) == 3) {
    std::vector<float> p(n * st);
    for (float& x : p)
      if (std::scanf("%f", &x) != 1) return 1;
    dg::Sum2 s(0.f);
    for (int q = 0; q < 4; ++q) s.add(dg::quarter_sum(p.data(), n, st, q));
    std::printf("%.17g ", s.wide());
    std::printf("%.17g\n", s.scale(k).wide());
  }
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    d = tmp_path_factory.mktemp("sum2")
    (d / "sum2.cpp").write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", os.path.join(ROOT, "paper_2502_09714_gb300", "csrc"),
                    str(d / "sum2.cpp"), "-o", str(d / "sum2")], check=True)
    return str(d / "sum2")


# modes of a face, rows of a plane and of an element, of the degrees 1 to 5
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5, 6, 9, 10, 15, 16, 21, 25, 36])
@pytest.mark.parametrize("st", [1, 2, 3])
def test_quarters(harness, n, st):
    rng = np.random.default_rng(100 * n + st)
    runs, text = [], []
    for _ in range(50):
        p = rng.normal(size=(n, st)) * 10.0 ** rng.uniform(-6, 6, size=(n, st))
        h = n // 2
        p[rng.permutation(n)[:h], 0] = -p[rng.permutation(n)[:h], 0]
        p = p.astype(np.float32)
        k = np.float32(rng.uniform(0.1, 1e4))
        runs.append((p[:, 0].astype(np.float64), float(k)))
        text.append(f"{n} {st} {k:.9g} " + " ".join(f"{x:.9g}" for x in p.ravel()))
    out = subprocess.run([harness], input="\n".join(text), capture_output=True, text=True, check=True).stdout.split()
    u = 2.0 ** -24
    for (x, k), s, sk in zip(runs, out[::2], out[1::2]):
        exact, mag = math.fsum(x), float(np.abs(x).sum())
        # each of the n + 3 additions adds an error of at most u times the partial sum to lo, exactly known, and
        # rounds lo itself once or twice
        tol = 2 * (n + 4) ** 2 * u * u * mag
        assert abs(float(s) - exact) <= tol
        assert abs(float(sk) - k * exact) <= k * (tol + 4 * u * u * (abs(exact) + (n + 4) * mag))
