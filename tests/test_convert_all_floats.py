"""The integer conversions (csrc/lorads_convert.h) against the casts where
test_convert_bits.py samples: every float widened, and every rounding boundary of the narrowing -- each
float's own value, the midpoint to the next one and the doubles beside that -- in the normal range and
one exponent beyond it at both ends."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2403_09133_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <thread>
#include <vector>
#include "lorads_convert.h"
static uint64_t bits(double x) { uint64_t b; memcpy(&b, &x, 8); return b; }
static uint32_t bits(float x) { uint32_t b; memcpy(&b, &x, 4); return b; }
static long run(uint32_t first, uint32_t last) {
  long bad = 0;
  for (uint64_t u = first; u < last; ++u) {
    uint32_t v = (uint32_t)u;
    float x; memcpy(&x, &v, 4);
    const double y = lorads::widen(x), z = (double)x;
    bad += x == x ? bits(y) != bits(z) : y == y;
    const uint32_t e = v >> 23 & 255u;
    if (v >> 31 || e == 0 || e == 255) continue;      // the narrowing: sign by sign below
    const uint64_t base = bits(z);
    const uint64_t at[4] = {base, base + 0xfffffffull, base + 0x10000000ull, base + 0x10000001ull};
    for (int k = 0; k < 4; ++k) {
      // both signs in turn: it is copied, not used
      const uint64_t b = at[k] | (uint64_t)(v & 1u) << 63;
      double d; memcpy(&d, &b, 8);
      bad += bits(lorads::narrow(d)) != bits((float)d);
    }
  }
  return bad;
}
int main() {
  const int n = 16;
  std::vector<std::thread> ts;
  std::vector<long> bad(n, 0);
  for (int i = 0; i < n; ++i)
    ts.emplace_back([&, i] {
      const uint64_t step = (1ull << 32) / n;
      bad[i] = run((uint32_t)(i * step), i + 1 == n ? 0xffffffffu : (uint32_t)((i + 1) * step));
    });
  long total = 0;
  for (int i = 0; i < n; ++i) { ts[i].join(); total += bad[i]; }
  // underflow, overflow and the ends of the normal range
  const double ends[] = {0x1p-126, 0x1.fffffep-127, 0x1.ffffffp-127, 0x1p-149, 0x1p-150, 0x1.8p-150,
                         0x1p-1074, 0x1.fffffep127, 0x1.fffffefffffffp127, 0x1.ffffffp127, 0x1p128,
                         0x1.fffffffffffffp1023, 0.0, INFINITY};
  for (double d : ends)
    for (double s : {d, -d}) total += bits(lorads::narrow(s)) != bits((float)s);
  std::printf("%ld\n", total);
  return total != 0;
}
"""


def test_every_float_and_rounding_boundary(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no g++")
    (tmp_path / "c.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O3", "-std=c++17", "-pthread", "-I", CSRC, str(tmp_path / "c.cpp"),
                    "-o", str(tmp_path / "c")], check=True)
    r = subprocess.run([str(tmp_path / "c")], capture_output=True, text=True)
    assert r.returncode == 0 and r.stdout.strip() == "0", r.stdout


DEVICE = r"""
#include "lorads_convert.h"
__global__ void k(unsigned long long* bad) {
  unsigned long long b = 0;
  const unsigned long long step = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long u = blockIdx.x * (unsigned long long)blockDim.x + threadIdx.x; u < 1ull << 32;
       u += step) {
    const float x = __uint_as_float((unsigned)u);
    const double y = lorads::widen(x), z = (double)x;
    b += x == x ? __double_as_longlong(y) != __double_as_longlong(z) : y == y;
    const unsigned e = (unsigned)u >> 23 & 255u;
    if (e == 0 || e == 255) continue;
    const unsigned long long off[4] = {0, 0xfffffffull, 0x10000000ull, 0x10000001ull};
    for (int i = 0; i < 4; ++i) {
      const double d = __longlong_as_double(__double_as_longlong(z) + off[i]);
      b += __float_as_uint(lorads::narrow(d)) != __float_as_uint((float)d);
    }
  }
  if (b) atomicAdd(bad, b);
}
extern "C" long long mismatches() {
  unsigned long long* d = nullptr;
  unsigned long long h = ~0ull;
  if (cudaMalloc(&d, 8) != cudaSuccess) return -1;
  cudaMemset(d, 0, 8);
  k<<<1216, 256>>>(d);
  const cudaError_t e = cudaMemcpy(&h, d, 8, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? (long long)h : -1;
}
"""


@pytest.mark.gpu
def test_every_float_on_the_device(cuda, tmp_path):
    """The device branch, whose bit patterns come from intrinsics."""
    import ctypes

    from paper_2403_09133_gb300 import build as B
    (tmp_path / "c.cu").write_text(DEVICE)
    lib = str(tmp_path / "c.so")
    subprocess.run([B.nvcc(), *B.ARCH, "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-shared", "-I",
                    CSRC, str(tmp_path / "c.cu"), "-o", lib], check=True)
    fn = ctypes.CDLL(lib).mismatches
    fn.restype = ctypes.c_longlong
    assert fn() == 0
