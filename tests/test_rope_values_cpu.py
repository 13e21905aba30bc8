"""The RoPE table's cosines and sines (a function of the CUDA sources that also compiles for the host) against the C
library's long double ones: good to the last bits of a double, so that rounding to fp32 is the only error, for every
angle that positions and frequencies give, those of a theta below 1 among them (CPU only; needs nvcc)."""
import subprocess

import pytest

from paper_2609_29029_gb300 import build

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include "rift_common.cuh"
int main() {
  // (positions, theta): a long context, and thetas below 1, whose frequencies grow to 1 / theta
  const double cases[4][2] = {{32768, 1e4}, {1e6, 1e6}, {2000, 1e-3}, {400, 1e-8}};
  for (auto& cs : cases) {
    long double worst = 0;
    double top = 0;
    for (int j = 0; j < 64; j += 7)
      for (double p = 0; p < cs[0]; p += cs[0] > 4000 ? 13 : 1) {
        const double x = p * std::pow(cs[1], -2.0 * j / 128);
        const double2 v = rift::rope_cos_sin_f64(x);
        worst = std::fmax(worst, std::fmax(std::fabs(v.x - cosl(x)), std::fabs(v.y - sinl(x))));
        top = std::fmax(top, x);
      }
    printf("%.3Lg %.3g\n", worst, top);
  }
}
"""


def test_cos_sin_are_good_to_a_doubles_last_bits(tmp_path):
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src = tmp_path / "rope.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "rope"
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-I", str(build.ROOT / "include"), "-I",
                    str(build.CSRC), *build.ARCH, str(src), "-o", str(exe)], check=True, capture_output=True)
    rows = [line.split() for line in subprocess.run([str(exe)], check=True, capture_output=True,
                                                    text=True).stdout.splitlines()]
    assert len(rows) == 4 and float(rows[3][1]) > 2.0 ** 32
    for worst, _ in rows:
        # two roundings of values up to 1 (2^-53 each) and of the reduced angle, the polynomials' 5e-17
        assert float(worst) < 3e-16, rows
