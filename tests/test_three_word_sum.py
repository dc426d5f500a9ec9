"""The sum over a warp's lanes in the double-float kernels (csrc/threeword.h), compiled for the host: 64
numbers hi + lo of random sizes and signs, added in the kernels' tree, against exact fractions. FP64 would
round the total at 2^-53 of the largest partial sum; held to that of the sum of absolute values
(two floats alone miss it by a factor of about 16)."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1501_01855_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include "threeword.h"
int main() {
  using ovl::ThreeWord;
  ThreeWord v[64];
  float h, l;
  int n = 0;
  while (scanf("%a %a", &h, &l) == 2) {
    v[n++] = ThreeWord{h, l, 0.f};
    if (n < 64) continue;
    for (int i = 0; i < 32; ++i) v[i] = v[i] + v[32 + i];   // the two numbers of a lane
    for (int o = 16; o > 0; o >>= 1)
      for (int i = 0; i < o; ++i) v[i] = v[i] + v[i + o];
    printf("%a\n", ovl::to_double(v[0]));
    n = 0;
  }
}
"""


def test_lane_sums_keep_fp64_accuracy(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src = tmp_path / "sum.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "sum")
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    rng = np.random.default_rng(4)
    rows = []
    for k in range(400):
        x = rng.standard_normal(64) ** 2 if k % 2 == 0 else rng.standard_normal(64) * np.exp(4 * rng.standard_normal(64))
        h = x.astype(np.float32)
        l = (x - h).astype(np.float32) * np.float32(1 + (k % 3))   # also low words that are not normalised
        rows.append((h, l))
    text = "".join("%s %s\n" % (float(a).hex(), float(b).hex()) for h, l in rows for a, b in zip(h, l))
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.split()
    assert len(out) == len(rows)
    for (h, l), got in zip(rows, out):
        terms = [Fraction(float(a)) + Fraction(float(b)) for a, b in zip(h, l)]
        assert abs(Fraction(float.fromhex(got)) - sum(terms)) <= Fraction(2) ** -53 * sum(abs(t) for t in terms)
