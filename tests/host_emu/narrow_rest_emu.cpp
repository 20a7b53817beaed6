// Host run of widen.cuh's narrow_rest (tests/test_narrow_rest_host.py) against the remainder formed
// in FP64: random values of |d| <= 1 over all exponents, ties of narrow, values next to powers of two.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>

static unsigned __float_as_uint(float f) { unsigned u; std::memcpy(&u, &f, 4); return u; }
static float __uint_as_float(unsigned u) { float f; std::memcpy(&f, &u, 4); return f; }
static int __double2hiint(double d) { uint64_t u; std::memcpy(&u, &d, 8); return (int)(u >> 32); }
static int __double2loint(double d) { uint64_t u; std::memcpy(&u, &d, 8); return (int)(uint32_t)u; }
static double __hiloint2double(int hi, int lo) {
  const uint64_t u = ((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo;
  double d;
  std::memcpy(&d, &u, 8);
  return d;
}
#include "widen_narrow.inc"

static long wrong = 0, runs = 0;
static void check(double d) {
  ++runs;
  const float got = narrow_rest(d);
  const float want = std::fabs(d) < 0x1p-74 ? 0.0f : narrow(d - widen(narrow(d)));
  if (got != want && wrong++ < 10) std::printf("%a: %a, not %a\n", d, got, want);
}

int main() {
  std::mt19937_64 rng(5);
  for (long i = 0; i < 4000000; ++i) {
    const uint64_t r = rng();
    const int e = i & 1 ? 0 : (int)((r >> 1) % 120);  // |d| in (0.5, 1], or down to 2^-120
    uint64_t man = rng() & 0xfffffffffffffull;
    if ((i & 6) == 2) man = (man & ~0x1fffffffull) | 0x10000000ull;                        // ties of narrow
    if ((i & 6) == 4) man = (man & ~0x1fffffffull) | (0x10000000ull + (r >> 61) - 4);      // next to them
    if ((i & 62) == 6) man = 0xfffffffffffffull - (r & 0x3fffffff);                        // a carry to the next power
    const uint64_t bits = (r & 0x8000000000000000ull) | (uint64_t)(1022 - e) << 52 | man;
    double d;
    std::memcpy(&d, &bits, 8);
    check(d);
  }
  for (double d : {0.0, -0.0, 1.0, -1.0, 0.5, 0x1p-74, 0x1.fffffffffffffp-75, 0x1.fffffffffffffp-1, 0x1p-1022, 0x1p-1074}) check(d);
  std::printf("%ld of %ld wrong\n", wrong, runs);
  return wrong != 0;
}
