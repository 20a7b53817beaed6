// Host run of the field's double-float complex product and phasor tables
// (tests/test_field_precision_host.py), their own text, against extended precision.
//   field_precision_emu cmul           -> rms and largest error of df::cmul, and of the double-float
//                                         products and sums it stands for (df::mul, df::add)
//   field_precision_emu phasors n M B  -> largest error of tab at the rows' last entries, and of
//                                         the split values' sums there
#define _GNU_SOURCE 1
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <vector>

struct dim3 {
  unsigned x = 1, y = 1, z = 1;
};
static dim3 blockIdx, threadIdx, blockDim, gridDim;
struct float4 { float x, y, z, w; };
struct double2 { double x, y; };
static float4 make_float4(float a, float b, float c, float d) { return {a, b, c, d}; }
static double2 make_double2(double a, double b) { return {a, b}; }
static int __double2hiint(double d) { uint64_t u; std::memcpy(&u, &d, 8); return (int)(u >> 32); }
static int __double2loint(double d) { uint64_t u; std::memcpy(&u, &d, 8); return (int)(uint32_t)u; }
static double __hiloint2double(int hi, int lo) {
  const uint64_t u = ((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo;
  double d;
  std::memcpy(&d, &u, 8);
  return d;
}
static unsigned __float_as_uint(float f) { unsigned u; std::memcpy(&u, &f, 4); return u; }
static float __uint_as_float(unsigned u) { float f; std::memcpy(&f, &u, 4); return f; }
static uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
#define MLMC_COV_EXP 1

#include "dfloat.cuh"

namespace mlmc {
#include "kernels.inc"
}  // namespace mlmc
using namespace mlmc;

static int run_cmul() {
  std::mt19937_64 rng(7);
  std::uniform_real_distribution<double> angle(-M_PI, M_PI);
  const long count = 2000000;
  double sq[2] = {}, top[2] = {};
  for (long i = 0; i < count; ++i) {
    const double t = angle(rng), u = angle(rng);
    const double v[4] = {std::cos(t), std::sin(t), std::cos(u), std::sin(u)};
    float h[4], l[4];
    for (int k = 0; k < 4; ++k) h[k] = (float)v[k], l[k] = (float)(v[k] - h[k]);
    const long double re = (long double)v[0] * v[2] - (long double)v[1] * v[3];
    const long double im = (long double)v[0] * v[3] + (long double)v[1] * v[2];
    float r[2][4], ah, al, bh, bl;
    df::cmul(h[0], l[0], h[1], l[1], h[2], l[2], h[3], l[3], r[0][0], r[0][1], r[0][2], r[0][3]);
    df::mul(h[0], l[0], h[2], l[2], ah, al);
    df::mul(h[1], l[1], h[3], l[3], bh, bl);
    df::add(ah, al, -bh, -bl, r[1][0], r[1][1]);
    df::mul(h[0], l[0], h[3], l[3], ah, al);
    df::mul(h[1], l[1], h[2], l[2], bh, bl);
    df::add(ah, al, bh, bl, r[1][2], r[1][3]);
    for (int k = 0; k < 2; ++k) {
      const double e1 = (double)fabsl((long double)r[k][0] + r[k][1] - re);
      const double e2 = (double)fabsl((long double)r[k][2] + r[k][3] - im);
      sq[k] += e1 * e1 + e2 * e2;
      top[k] = std::max(top[k], std::max(e1, e2));
    }
  }
  std::printf("%.6e %.6e %.6e %.6e\n", std::sqrt(sq[0] / (2 * count)), top[0], std::sqrt(sq[1] / (2 * count)), top[1]);
  return 0;
}

static int run_phasors(int n, int M, int B) {
  std::mt19937_64 rng(11);
  std::normal_distribution<double> normal(0.0, 10.0);
  std::vector<double> w((size_t)B * M * 3), b((size_t)B * M);
  for (double& v : w) v = normal(rng);
  for (double& v : b) v = std::fabs(normal(rng));
  std::vector<double2> tab((size_t)B * 3 * M * n);
  std::vector<float4> xs(tab.size());
  const double h = 1.0 / (n - 1);
  gridDim = dim3{64, 1, 1};
  blockDim = dim3{1, 1, 1};
  for (unsigned t = 0; t < gridDim.x; ++t) {
    blockIdx.x = t;
    threadIdx.x = 0;
    k_phasors(w.data(), b.data(), B, M, n, h, tab.data(), xs.data());
  }
  double last = 0.0, split = 0.0;
  for (int s = 0; s < B; ++s)
    for (int a = 0; a < 3; ++a)
      for (int m = 0; m < M; ++m) {
        const size_t o = (((size_t)s * 3 + a) * M + m) * n + n - 1, f = (size_t)s * M + m;
        double ph = w[3 * f + a] * ((double)(n - 1) * h);  // the phase as the table defines it
        if (a == 0) ph += b[f];
        const long double c = cosl((long double)ph), q = sinl((long double)ph);
        last = std::max(last, (double)std::max(fabsl(tab[o].x - c), fabsl(tab[o].y - q)));
        split = std::max(split, (double)std::max(fabsl((long double)xs[o].x + xs[o].y - c),
                                                 fabsl((long double)xs[o].z + xs[o].w - q)));
      }
  std::printf("%.6e %.6e\n", last, split);
  return 0;
}

int main(int argc, char** argv) {
  if (argc == 2 && !std::strcmp(argv[1], "cmul")) return run_cmul();
  if (argc == 5) return run_phasors(std::atoi(argv[2]), std::atoi(argv[3]), std::atoi(argv[4]));
  return 2;
}
