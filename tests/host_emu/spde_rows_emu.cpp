// Host run of the SPDE correction cycle's kernels as the library launches them
// (tests/test_spde_rows_host.py): the row-of-four colour passes, the red restriction, the black
// interpolation and the one-block cycle of the small grids, their own text, against the plain
// one-cell forms, and a whole field through them.
//   spde_rows_emu check                                  -> "ok" or what differs
//   spde_rows_emu field seed id n n_noise sigma2 ell     -> k at the n^3 nodes (hex doubles)
#define _GNU_SOURCE 1
#include <algorithm>
#include <barrier>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <random>
#include <thread>
#include <vector>

#include "mlmc.h"

struct dim3 {
  unsigned x = 1, y = 1, z = 1;
  dim3(unsigned a = 1, unsigned b = 1, unsigned c = 1) : x(a), y(b), z(c) {}
};
static thread_local dim3 blockIdx, threadIdx;
static dim3 blockDim, gridDim;
using std::min;

static unsigned __float_as_uint(float f) { unsigned u; std::memcpy(&u, &f, 4); return u; }
static float __uint_as_float(unsigned u) { float f; std::memcpy(&f, &u, 4); return f; }
static float __fmul_rn(float a, float b) { return a * b; }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fdiv_rn(float a, float b) { return a / b; }
static float __fsqrt_rn(float a) { return std::sqrt(a); }
static float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static uint32_t __umulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
static int __double2hiint(double d) { uint64_t b; std::memcpy(&b, &d, 8); return (int)(uint32_t)(b >> 32); }
static int __double2loint(double d) { uint64_t b; std::memcpy(&b, &d, 8); return (int)(uint32_t)b; }
static double __hiloint2double(int hi, int lo) {
  uint64_t b = ((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo;
  double d;
  std::memcpy(&d, &b, 8);
  return d;
}
struct float2 { float x, y; };
struct alignas(16) float4 { float x, y, z, w; };
static float2 make_float2(float a, float b) { return {a, b}; }
static float4 make_float4(float a, float b, float c, float d) { return {a, b, c, d}; }
static std::barrier<>* block_barrier = nullptr;
static void __syncthreads() { block_barrier->arrive_and_wait(); }
static int __popc(unsigned v) { return __builtin_popcount(v); }
static int atomicOr(int* p, int v) {
  const int o = *p;
  *p |= v;
  return o;
}

// block reduction stand-in: the threads of a block run from the last to thread 0
static double g_block_acc = 0.0;
template <int THREADS>
static double block_sum(double v) {
  if (threadIdx.x == blockDim.x - 1) g_block_acc = 0.0;
  g_block_acc += v;
  return g_block_acc;
}
static double warp_partial_sum(const double* part, int NB) {
  double a = 0.0;
  for (int b = 0; b < NB; ++b) a += part[b];
  return a;
}

#include "spde_kernels.inc"

template <typename F>
static void launch(dim3 grid, dim3 block, F body) {
  gridDim = grid;
  blockDim = block;
  for (unsigned bz = 0; bz < grid.z; ++bz)
    for (unsigned by = 0; by < grid.y; ++by)
      for (unsigned bx = 0; bx < grid.x; ++bx)
        for (int t = (int)block.x - 1; t >= 0; --t) {
          blockIdx = dim3(bx, by, bz);
          threadIdx = dim3((unsigned)t, 0, 0);
          body();
        }
}


using Vec = std::vector<float>;
struct Diag {
  float ch2, i3, i4, i5, i6;
  explicit Diag(double c) : ch2((float)c), i3((float)(1.0 / (c + 3.0))), i4((float)(1.0 / (c + 4.0))), i5((float)(1.0 / (c + 5.0))), i6((float)(1.0 / (c + 6.0))) {}
};

// the one-block kernel with its threads as threads
static void run_tail(int lc, const TailDiag& td, const float* g, float* e, const int* active, int samples) {
  std::barrier<> bar(kTailThreads);
  block_barrier = &bar;
  for (int s = 0; s < samples; ++s) {
    std::vector<std::thread> th;
    for (int t = 0; t < kTailThreads; ++t)
      th.emplace_back([&, t] {
        blockIdx = dim3((unsigned)s, 0, 0);
        threadIdx = dim3((unsigned)t, 0, 0);
        if (active[s]) k_cc_tail(lc, td, g, e, active);
      });
    for (auto& x : th) x.join();
  }
}

static TailDiag tail_diag(int lc, double ch2_finest) {
  TailDiag td{};
  double c = ch2_finest;
  for (int k = lc; k >= 1; --k, c *= 4.0) {
    td.ch2[k] = (float)c;
    for (int np = 3; np <= 6; ++np) td.inv[k][np - 3] = (float)(1.0 / (c + (double)np));
  }
  return td;
}

static int wrong = 0;
static void report(bool ok, const char* what, int lc, double c) {
  if (!ok && wrong++ < 20) std::printf("%s, C = %d, c h^2 = %g\n", what, 1 << lc, c);
}
static int colour_of(size_t q, int lc) {
  const size_t m = ((size_t)1 << lc) - 1;
  return (int)(((q & m) + ((q >> lc) & m) + (q >> (2 * lc))) & 1);
}

static void check_grid(int lc, double c, int B, std::mt19937& rng) {
  const int C = 1 << lc;
  const size_t C3 = (size_t)C * C * C, cells = B * C3;
  const Diag d(c);
  std::uniform_real_distribution<float> U(-1.0f, 1.0f);
  Vec g(cells), Z(cells);
  for (float& v : g) v = U(rng);
  for (float& v : Z) v = U(rng);
  std::vector<int> active(B, 1);
  active[1] = 0;  // a finished sample keeps its values
  const dim3 quads = cell_grid(C3 / 4, B), half = cell_grid(C3 / 2, B);
  for (int colour = 0; colour < 2; ++colour) {
    Vec a = Z, b = Z;
    launch(half, dim3(kT), [&] { k_cc_rbgs<float>(colour, lc, B, d.i3, d.i4, d.i5, d.i6, g.data(), a.data(), active.data()); });
    launch(quads, dim3(kT), [&] { k_cc_rbgs4<false>(colour, lc, B, d.i3, d.i4, d.i5, d.i6, g.data(), b.data(), active.data()); });
    report(a == b, colour ? "black pass" : "red pass", lc, c);
  }
  {
    Vec a(cells, 0.0f), b = Z;
    launch(half, dim3(kT), [&] { k_cc_rbgs<float>(0, lc, B, d.i3, d.i4, d.i5, d.i6, g.data(), a.data(), active.data()); });
    launch(quads, dim3(kT), [&] { k_cc_rbgs4<true>(0, lc, B, d.i3, d.i4, d.i5, d.i6, g.data(), b.data(), active.data()); });
    bool ok = true;
    for (size_t q = 0; q < cells; ++q) {
      const bool hit = active[q / C3] && !colour_of(q % C3, lc);
      ok = ok && b[q] == (hit ? a[q] : Z[q]);
    }
    report(ok, "red pass from zero", lc, c);
  }
  if (lc < 2) return;
  const int Cc = C / 2;
  const size_t Cc3 = C3 / 8;
  {
    Vec r(cells, 0.0f), full(B * Cc3, -7.0f), red(B * Cc3, -7.0f);
    int zs = 0;
    const int slabs = zslabs(C, &zs);
    launch(dim3(col_blocks(C), slabs, B), dim3(128), [&] {
      k_cc_residual<float, float>(lc, zs, d.ch2, g.data(), Z.data(), r.data(), nullptr, active.data());
    });
    for (size_t q = 0; q < cells; ++q)
      if (colour_of(q % C3, lc)) r[q] = 0.0f;
    launch(cell_grid(Cc3, B), dim3(kT), [&] { k_cc_restrict<float>(lc - 1, B, r.data(), full.data(), active.data()); });
    launch(cell_grid(Cc3 / 2, B), dim3(kT), [&] {
      k_cc_restrict_red(lc, B, d.ch2, g.data(), Z.data(), red.data(), active.data());
    });
    // both add four residuals of values up to 1 + (c h^2 + 12): nine roundings each
    const float tol = 0.5f * 4.0f * 9.0f * (13.0f + d.ch2) * 0x1p-24f;
    bool ok = true;
    for (size_t q = 0; q < full.size(); ++q) ok = ok && std::fabs(full[q] - red[q]) <= tol && (active[q / Cc3] || red[q] == -7.0f);
    report(ok, "red restriction", lc, c);
  }
  {
    Vec e(B * Cc3), a = Z, b = Z;
    for (float& v : e) v = U(rng);
    launch(cell_grid(C3, B), dim3(kT), [&] { k_cc_prolong<float>(lc, B, e.data(), a.data(), active.data()); });
    launch(quads, dim3(kT), [&] { k_cc_prolong_black(lc, B, e.data(), b.data(), active.data()); });
    bool ok = true;
    for (size_t q = 0; q < cells; ++q) ok = ok && b[q] == (colour_of(q % C3, lc) ? a[q] : Z[q]);
    report(ok, "black interpolation", lc, c);
  }
}

// One V(2,2) cycle from a zero guess by the row kernels down to the 2^3 grid (one cell per thread).
static void rows_cycle(int lc, double c, int B, const Vec& g, Vec& e, const int* active) {
  const int C = 1 << lc;
  const size_t C3 = (size_t)C * C * C;
  const Diag d(c);
  if (lc == 1) {
    launch(dim3(1), dim3(128), [&] { k_cc_coarse<float>(B, d.ch2, g.data(), e.data(), active); });
    return;
  }
  const dim3 quads = cell_grid(C3 / 4, B);
  auto pass = [&](int colour, bool zero) {
    launch(quads, dim3(kT), [&] {
      if (zero) k_cc_rbgs4<true>(colour, lc, B, d.i3, d.i4, d.i5, d.i6, g.data(), e.data(), active);
      else k_cc_rbgs4<false>(colour, lc, B, d.i3, d.i4, d.i5, d.i6, g.data(), e.data(), active);
    });
  };
  pass(0, true), pass(1, false), pass(0, false), pass(1, false);
  Vec gc(B * C3 / 8, 0.0f), ec(B * C3 / 8, 0.0f);
  launch(cell_grid(C3 / 16, B), dim3(kT), [&] { k_cc_restrict_red(lc, B, d.ch2, g.data(), e.data(), gc.data(), active); });
  rows_cycle(lc - 1, 4.0 * c, B, gc, ec, active);
  launch(quads, dim3(kT), [&] { k_cc_prolong_black(lc, B, ec.data(), e.data(), active); });
  pass(0, false), pass(1, false), pass(0, false), pass(1, false);
}

static void check_tail(int lc, double c, std::mt19937& rng) {
  const size_t C3 = (size_t)1 << (3 * lc);
  const int B = 2;
  std::uniform_real_distribution<float> U(-1.0f, 1.0f);
  Vec g(B * C3), a(B * C3, 5.0f), b(B * C3, 5.0f);
  for (float& v : g) v = U(rng);
  const int active[2] = {1, 1};
  rows_cycle(lc, c, B, g, a, active);
  run_tail(lc, tail_diag(lc, c), g.data(), b.data(), active, B);
  report(a == b, "one-block cycle", lc, c);
}

// The cycle as the library runs it: rows above kTailC cells per axis, one block from there.
static void cycle(int lc, double c, const Vec& g, Vec& e, const int* active) {
  const int C = 1 << lc;
  if (C <= kTailC) {
    run_tail(lc, tail_diag(lc, c), g.data(), e.data(), active, 1);
    return;
  }
  const size_t C3 = (size_t)C * C * C;
  const Diag d(c);
  const dim3 quads = cell_grid(C3 / 4, 1);
  auto pass = [&](int colour, bool zero) {
    launch(quads, dim3(kT), [&] {
      if (zero) k_cc_rbgs4<true>(colour, lc, 1, d.i3, d.i4, d.i5, d.i6, g.data(), e.data(), active);
      else k_cc_rbgs4<false>(colour, lc, 1, d.i3, d.i4, d.i5, d.i6, g.data(), e.data(), active);
    });
  };
  pass(0, true), pass(1, false), pass(0, false), pass(1, false);
  Vec gc(C3 / 8), ec(C3 / 8);
  launch(cell_grid(C3 / 16, 1), dim3(kT), [&] { k_cc_restrict_red(lc, 1, d.ch2, g.data(), e.data(), gc.data(), active); });
  cycle(lc - 1, 4.0 * c, gc, ec, active);
  launch(quads, dim3(kT), [&] { k_cc_prolong_black(lc, 1, ec.data(), e.data(), active); });
  pass(0, false), pass(1, false), pass(0, false), pass(1, false);
}

static int field(char** argv) {
  const uint64_t seed = std::strtoull(argv[1], nullptr, 10), id = std::strtoull(argv[2], nullptr, 10);
  const int n = std::atoi(argv[3]), n_noise = std::atoi(argv[4]);
  const double sigma2 = std::atof(argv[5]), ell = std::atof(argv[6]);
  const int C = 2 * (n - 1), lc = log2i(C), r = (n_noise - 1) / (n - 1);
  const size_t C3 = (size_t)C * C * C;
  const double h = 1.0 / (double)(n - 1), hf = 1.0 / (double)(n_noise - 1), v = 0.5 * hf;
  const double scale = std::sqrt(v * v * v) / h;
  const uint64_t Mo = 4 * (uint64_t)(n_noise - 1) + 1;
  std::vector<double> g64(C3), Z64(C3, 0.0);
  uint64_t ids[1] = {id};
  launch(cell_grid(C3, 1), dim3(kT), [&] {
    k_spde_noise(ids, 1, lc, r, Mo, (uint32_t)seed, (uint32_t)(seed >> 32), scale, g64.data());
  });
  Vec g32(C3), e32(C3);
  int active[1] = {1}, cycles[1] = {0}, flag = 0;
  int zs = 0;
  const int slabs = zslabs(C, &zs), NB = col_blocks(C) * slabs;
  std::vector<double> partial(NB), g2(1);
  launch(dim3(col_blocks(C), slabs, 1), dim3(128), [&] {
    k_cc_residual<double, float>(lc, zs, 0.0, g64.data(), nullptr, nullptr, partial.data(), active);
  });
  launch(dim3(1), dim3(128), [&] { k_cc_sum(1, NB, partial.data(), g2.data(), active); });
  const double kappa = 1.0 / ell, ch2 = kappa * kappa * h * h;
  for (int c = 0; c <= kSpdeMaxCycles; ++c) {
    launch(dim3(col_blocks(C), slabs, 1), dim3(128), [&] {
      k_cc_residual64(lc, zs, ch2 + 3.0, ch2 + 4.0, ch2 + 5.0, ch2 + 6.0, g64.data(), Z64.data(), g32.data(),
                      partial.data(), active);
    });
    flag = 0;
    launch(dim3(1), dim3(128), [&] {
      k_cc_check(1, NB, c, partial.data(), g2.data(), kSpdeRtol, kSpdeMaxCycles, active, cycles, &flag);
    });
    if (!(flag & 1)) break;
    cycle(lc, ch2, g32, e32, active);
    launch(cell_grid(C3, 1), dim3(kT), [&] { k_cc_update(lc, 1, e32.data(), Z64.data(), active); });
  }
  std::fprintf(stderr, "cycles %d flag %d\n", cycles[0], flag);
  const int off = (n - 1) / 2;
  const double a = std::sqrt(8.0 * 3.14159265358979323846 * kappa * sigma2);
  const size_t nodes = (size_t)n * n * n;
  std::vector<double> k(nodes);
  launch(dim3((unsigned)((nodes + kT - 1) / kT)), dim3(kT), [&] {
    k_spde_extract(n, C, off, 1, a, Z64.data(), MLMC_F64, k.data());
  });
  for (double x : k) {
    uint64_t b;
    std::memcpy(&b, &x, 8);
    std::printf("%016llx\n", (unsigned long long)b);
  }
  return (flag & 2) ? 2 : 0;
}

int main(int argc, char** argv) {
  if (argc == 8) return field(argv + 1);
  std::mt19937 rng(3);
  for (double c : {0.0, 1e-4, 0.3, 40.0}) {
    for (int lc : {2, 3, 4, 5}) check_grid(lc, c, 3, rng);
    if (c > 0.0)  // (the 2^3 solve needs c h^2 > 0)
      for (int lc : {2, 3, 4}) check_tail(lc, c, rng);
  }
  if (!wrong) std::printf("ok\n");
  return wrong ? 1 : 0;
}
