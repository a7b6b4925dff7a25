"""quotient_by (csrc/quotient.h) against the device's division, bit for bit: random dividends of every
exponent down to 2^-900 and divisors over the range that quotient_ok admits, and divisors of all ones and
one above a power of two, where a reciprocal is at its worst."""
import os
import shutil
import subprocess

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SRC = r"""
#include <cstdio>
#include <cstdint>
#include <cuda_runtime.h>
#include "quotient.h"
__device__ uint64_t mix(uint64_t x) {  // splitmix64
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}
__device__ double number(uint64_t bits, int lo, int hi) {  // mantissa of the low bits, exponent in [lo, hi]
  const uint64_t e = 1023 + lo + int((bits >> 52) % uint64_t(hi - lo + 1));
  return __longlong_as_double((long long)((e << 52) | (bits & 0xfffffffffffffull)));
}
__global__ void k(unsigned long long* bad, unsigned long long* done) {
  const uint64_t t = blockIdx.x * uint64_t(blockDim.x) + threadIdx.x;
  for (int i = 0; i < 64; ++i) {
    const uint64_t a = mix(3 * (64 * t + i)), b = mix(3 * (64 * t + i) + 1), c = mix(3 * (64 * t + i) + 2);
    double d = number(a, i % 2 ? -900 : -8, i % 2 ? 899 : 8);
    if (i % 16 == 3) d = __longlong_as_double(__double_as_longlong(d) | 0xfffffffffffffll);
    if (i % 16 == 7) d = __longlong_as_double((__double_as_longlong(d) & ~0xfffffffffffffll) | 1ll);
    const int top = int((__double_as_longlong(d) >> 52) & 2047) - 1023;
    const int low = top - 60 * int(c % 8);
    double v = number(b, low < -900 ? -900 : low, top);
    if (c & 16) v = -v;
    if (fabs(v) > d) v *= 0.5;
    if (fabs(v) < 0x1p-900 || !gdsw::quotient_ok(d)) continue;
    atomicAdd(done, 1ull);
    if (__double_as_longlong(gdsw::quotient_by(v, d, 1.0 / d)) != __double_as_longlong(v / d)) atomicAdd(bad, 1ull);
  }
}
int main() {
  unsigned long long *p, h[2];
  if (cudaMalloc(&p, 16) != cudaSuccess || cudaMemset(p, 0, 16) != cudaSuccess) return 2;
  k<<<4096, 256>>>(p, p + 1);
  if (cudaMemcpy(h, p, 16, cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  printf("%llu %llu\n", h[0], h[1]);
  return 0;
}
"""


def test_quotients_round_like_the_division(tmp_path):
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    csrc = os.path.join(os.path.dirname(__file__), "..", "paper_2606_01433_gb300", "csrc")
    (tmp_path / "q.cu").write_text(SRC)
    exe = str(tmp_path / "q")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-I", csrc, "-o", exe,
                    str(tmp_path / "q.cu")], check=True, timeout=300)
    out = subprocess.run([exe], check=True, timeout=120, capture_output=True, text=True).stdout.split()
    bad, done = int(out[0]), int(out[1])
    assert done > 60_000_000 and bad == 0
