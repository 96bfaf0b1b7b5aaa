"""The scale of a correction's columns and their fixed-point digits (csrc/refine_fixed.cuh), compiled for the host."""
import subprocess

import pytest

SOURCE = r"""
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include "refine_fixed.cuh"
using namespace mps;

// the value that 7 balanced digits of x at scale 2^e stand for
static double digits(float x, int e) {
  const uint64_t q = oz_fixed(x, e);
  double v = 0.0;
  for (int b = 6; b >= 0; --b) v = v * 256.0 + (double)((int)(q >> (8 * b) & 0xff) - 128);
  return std::ldexp(v, e - 54);
}

int main() {
  int bad = 0, n = 0;
  srand(5);
  auto uniform = [] { return (float)(rand() / (RAND_MAX + 1.0)); };
  for (int trial = 0; trial < 20000; ++trial) {
    // a column of up to 40 entries at one size, the diagonal at and just below a power of two, of either sign
    const int K = 1 + rand() % 40, size = -(rand() % 24), shift = rand() % 3 - 1, own = rand() % K;
    float x[40], y[40];
    CorrectionScale cs;
    for (int k = 0; k < K; ++k) {
      x[k] = std::ldexp(2 * uniform() - 1, size);
      y[k] = std::ldexp(2 * uniform() - 1, size);
      if (k == own) {
        x[k] = std::ldexp(1.f - std::ldexp(uniform(), -(rand() % 24)), size) * (rand() % 3 ? -1.f : 1.f);
        y[k] = 0.f;
      }
      cs.add(x[k], y[k], 0, shift, k == own);
    }
    const int e = cs.scale(shift) - shift;
    x[own] += cs.second_order();
    for (int k = 0; k < K; ++k)
      for (float v : {x[k], y[k]}) {
        ++n;
        if (!(std::fabs(v) < std::ldexp(1.0, e))) ++bad;
        if (std::fabs(digits(v, e) - (double)v) > std::ldexp(0.5, e - 54)) ++bad;
      }
  }
  std::printf("%d %d\n", n, bad);
  return bad != 0;
}
"""


@pytest.mark.slow
def test_every_part_of_a_column_lies_below_its_scale(tmp_path):
    """|x| < 2^e for every part, the diagonal with its second-order part included, and the digits give x back to
    half a unit of 2^(e - 54)."""
    import __graft_entry__ as g
    b = g._build_module()
    src, exe = tmp_path / "scale.cu", tmp_path / "scale"
    src.write_text(SOURCE)
    subprocess.run([b.nvcc(), *b.ARCH, "-std=c++17", "-I", b.SRC, str(src), "-o", str(exe)], check=True, capture_output=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
