"""The solver's integer float/double conversions (csrc/lorads_convert.h) against the casts, bit for
bit: every exponent of both formats with edge and random fractions, ties, zeros, subnormals,
overflow, infinities and NaN, compiled for the host."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2403_09133_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "lorads_convert.h"
static uint64_t bits(double x) { uint64_t b; memcpy(&b, &x, 8); return b; }
static uint32_t bits(float x) { uint32_t b; memcpy(&b, &x, 4); return b; }
int main() {
  std::mt19937_64 g(7);
  long bad = 0, n = 0;
  for (uint32_t s = 0; s < 2; ++s)
    for (uint32_t e = 0; e < 256; ++e)
      for (int k = 0; k < 4096; ++k) {
        const uint32_t m = k == 0 ? 0u : k == 1 ? 1u : k == 2 ? 0x7fffffu : (uint32_t)g() & 0x7fffffu;
        const uint32_t u = s << 31 | e << 23 | m;
        float x; memcpy(&x, &u, 4);
        const double y = lorads::widen(x), z = (double)x;
        ++n;
        if (std::isnan(x) ? !std::isnan(y) : bits(y) != bits(z)) ++bad;
      }
  for (uint64_t s = 0; s < 2; ++s)
    for (uint64_t e = 0; e < 2048; ++e)
      for (int k = 0; k < 1024; ++k) {
        uint64_t m = g() & 0xfffffffffffffull;
        // the dropped 29 bits at their edges: 0, 1, half - 1, half, half + 1, all; both parities
        const uint64_t low[6] = {0, 1, 0xfffffff, 0x10000000, 0x10000001, 0x1fffffff};
        if (k < 600) m = (m & ~0x1fffffffull) | low[k % 6];
        if (k < 12) m = (k < 6 ? 0xfffffe0000000ull : 0ull) | low[k % 6];
        const uint64_t b = s << 63 | e << 52 | m;
        double x; memcpy(&x, &b, 8);
        const float y = lorads::narrow(x), z = (float)x;
        ++n;
        if (std::isnan(x) ? !std::isnan(y) : bits(y) != bits(z)) ++bad;
      }
  std::printf("%ld %ld\n", n, bad);
  return bad != 0;
}
"""


def test_conversions_equal_the_casts(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    src = tmp_path / "convert.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "convert"
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    n, bad = map(int, r.stdout.split())
    assert n == 2 * 256 * 4096 + 2 * 2048 * 1024 and bad == 0
