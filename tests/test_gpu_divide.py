"""The operator set-up's short FP64 quotients (csrc/divide.cuh) against the language's division, on the
GPU, by a small program built here: random operands over all exponents (so both sides of every limit
of the short form), operands next to its limits and next to powers of two, zeros, infinities, NaN
and subnormal numbers. A quotient may differ only where the exact one is next to a tie, within 2^-30 of
an ulp (its remainders against the two neighbours are opposite up to that), and by one ulp; harmonic
means and reciprocals the same."""
import os
import subprocess

import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1607_03252_gb300", "csrc")

SOURCE = r"""
#include <cstdint>
#include <cstdio>
#include "divide.cuh"
using namespace mlmc;

__device__ uint64_t mix(uint64_t x) {  // splitmix64
  x += 0x9e3779b97f4a7c15ull;
  x = (x ^ (x >> 30)) * 0xbf58476d1ce4e5b9ull;
  x = (x ^ (x >> 27)) * 0x94d049bb133111ebull;
  return x ^ (x >> 31);
}
__device__ double any(uint64_t r, int mode) {  // mode 0: all bits; 1: exponent within 8 of 1; 2: near the limits
  if (mode == 0) return __longlong_as_double((long long)r);
  const uint64_t sign = r & 0x8000000000000000ull, man = r & 0xfffffffffffffull;
  const int pick = (int)(mix(r) & 15);
  const uint64_t e = mode == 1 ? 1015 + pick : (pick < 8 ? 919 + pick : 1119 + pick);
  const uint64_t m = (mix(r + 1) & 7) == 0 ? (man & 3) : ((mix(r + 1) & 7) == 1 ? 0xfffffffffffffull - (man & 3) : man);
  return __longlong_as_double((long long)(sign | e << 52 | m));
}
__device__ bool same(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b) || (isnan(a) && isnan(b));
}
// a and b are neighbours and n / d lies between them next to the middle
__device__ bool next_to_tie(double n, double d, double a, double b) {
  const long long u = __double_as_longlong(a) - __double_as_longlong(b);
  const double ra = fma(-d, a, n), rb = fma(-d, b, n);
  return (u == 1 || u == -1) && fabs(ra + rb) <= 0x1p-30 * fabs(ra);
}
__device__ int wrong(double n, double d) {
  const double m = __dmul_rn(2.0 * n, d), s = __dadd_rn(n, d);
  const double num[3] = {n, 1.0, m}, den[3] = {d, d, s};
  const double got[3] = {divide(n, d), reciprocal(d), harmonic(n, d)};
  int bad = 0;
  for (int q = 0; q < 3; ++q) {
    const double want = __ddiv_rn(num[q], den[q]);
    bad += !same(got[q], want) && !next_to_tie(num[q], den[q], got[q], want);
  }
  return bad;
}
__global__ void check(uint64_t seed, int mode, int per, unsigned long long* count) {
  const uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int i = 0; i < per; ++i) {
    const uint64_t k = mix(seed + t * (uint64_t)per + i);
    const double n = any(k, mode), d = any(mix(k), mode);
    if (const int bad = wrong(n, d)) atomicAdd(count, (unsigned long long)bad);
  }
}
__global__ void special(unsigned long long* count) {
  const double v[] = {0.0, -0.0, 1.0, -1.0, 3.0, 0x1p-1074, 0x1p-1022, 0x1p-101, 0x1p-100, 0x1.fffffffffffffp100, 0x1p101,
                      0x1.fffffffffffffp1023, INFINITY, -INFINITY, NAN};
  const int m = sizeof(v) / sizeof(v[0]);
  const int i = threadIdx.x / m, j = threadIdx.x % m;
  if (i >= m) return;
  if (const int bad = wrong(v[i], v[j])) atomicAdd(count, (unsigned long long)bad);
}
int main() {
  unsigned long long *count, host = 0;
  if (cudaMalloc(&count, sizeof(host)) != cudaSuccess || cudaMemset(count, 0, sizeof(host)) != cudaSuccess) return 2;
  for (int mode = 0; mode < 3; ++mode) check<<<1024, 256>>>(1000 + mode, mode, 128, count);
  special<<<1, 256>>>(count);
  if (cudaMemcpy(&host, count, sizeof(host), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  std::printf("%llu\n", host);
  return 0;
}
"""


def test_quotients_are_the_language_s(tmp_path):
    from paper_1607_03252_gb300.build import ARCH, nvcc

    (tmp_path / "check.cu").write_text(SOURCE)
    exe = tmp_path / "check"
    res = subprocess.run([nvcc(), *ARCH, "-O3", "-std=c++17", "-I", CSRC, str(tmp_path / "check.cu"), "-o", str(exe)],
                         capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stderr[-4000:]
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0, (res.returncode, res.stdout)
    assert int(res.stdout) == 0  # of 3 * 10^8
