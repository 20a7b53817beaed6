// Batched geometric multigrid: V(nu1, nu2) cycles with red-black Gauss-Seidel, full
// weighting, trilinear prolongation, rediscretised coarse operators and an exact 5^3
// solve (the deterministic solver inside every sample of Algorithm 1, for the model problem
// of Sec. 3, Eq. 16; the cycle family of Sec. 7.1).
//
// Scaled form. With faces K_pq = 2 k_p k_q / (k_p + k_q) and D_p = sum_q K_pq, every
// grid stores the h^2-scaled operator (A~ u)_p = D_p u_p - sum_q K_pq u_q and the
// scaled right-hand side g = h^2 f, so
//   smoothing     u_p <- (g_p + sum_q K_pq u_q) * (1 / D_p)      (6 FMA + 1 MUL)
//   residual      r~_p = g_p - D_p u_p + sum_q K_pq u_q = h^2 r_p  (7 FMA)
//   restriction   g_c = h_c^2 FW(r) = 4 FW(r~)
//   norms         ||r|| / ||f|| = ||r~|| / ||g||.
// No division runs inside a cycle; faces, D and 1/D are computed once per solve.
//
// Precision MLMC_PREC_MIXED: the V-cycle's faces are the FP32 harmonic means of the
// FP32-rounded nodal k and the V-cycle runs entirely in FP32 as a correction solve; the
// outer residual g - A~ u, on FP64 faces of the FP64 nodal k of the finest grid, and the
// update u += e run in FP64 (iterative refinement, or flexible CG with the FP32 cycle as
// preconditioner): the fixed point is the FP64 solution of the FP64 operator, the one
// an all-FP64 solve reaches.
//
// Every kernel skips samples whose `active` flag is 0, so each sample stops at its own
// cycle count; every per-sample sum is a fixed tree that depends only on n. A sample's
// result therefore does not depend on the batch it is solved in.
#include <math.h>
#include <stdio.h>
#include <stdlib.h>

#include <shared_mutex>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "divide.cuh"
#include "mg.cuh"
#include "optin.cuh"
#include "prof.cuh"
#include "smooth.cuh"
#include "tune.cuh"
#include "widen.cuh"

namespace mlmc {

namespace {

constexpr int kThreads = 256;
constexpr int kMaxLevels = 12;
constexpr int kPlaneThreads = 128;
constexpr int kCtaMaxN = 33;  // largest grid of the small-grid engine

// Plane launches: blockIdx.x (with threadIdx.x) enumerates the work items of one z-plane,
// blockIdx.y strides over the (sample, z) planes, so every in-sample index is 32-bit
// (n^3 < 2^31 for every valid n) and no thread divides a 64-bit index.
inline dim3 plane_grid(int per_plane, long long planes) {
  return dim3((unsigned)((per_plane + kPlaneThreads - 1) / kPlaneThreads),
              (unsigned)(planes < 65535 ? (planes > 0 ? planes : 1) : 65535));
}

size_t a256(size_t b) { return (b + 255) & ~(size_t)255; }

// Colour-split storage (see the colour-split kernels below).
__host__ __device__ __forceinline__ int split_pitch(int n) { return (((n + 1) >> 1) + 3) & ~3; }
// elements of one sample in colour-split storage
__host__ __device__ __forceinline__ size_t split_elems(int n) { return (size_t)2 * n * n * (size_t)split_pitch(n); }
__device__ __forceinline__ unsigned split_index(int n, int x, int y, int z) {
  const int P = split_pitch(n);
  return (unsigned)((x + y + z) & 1) * (unsigned)(n * n * P) + (unsigned)((z * n + y) * P + (x >> 1));
}

// Index of node (x, y, z) of sample s of an n^3 grid in the plain or (SPLIT) the
// colour-split storage.
template <bool SPLIT>
__device__ __forceinline__ size_t node_at(int n, int s, int x, int y, int z) {
  return SPLIT ? (size_t)s * split_elems(n) + split_index(n, x, y, z)
               : (((size_t)s * n + z) * n + y) * n + x;
}

// Carves 256-byte aligned pieces; with base == nullptr it only measures.
struct Carver {
  char* base;
  size_t off = 0;
  explicit Carver(void* b) : base((char*)b) {}
  template <typename T>
  T* take(size_t count) {
    T* p = base ? (T*)(base + off) : nullptr;
    off += a256(count * sizeof(T)) + 256;  // slack: 16-byte-rounded bulk copies may read past the end
    return p;
  }
};

// x in the arithmetic type TD (FP32 to FP64 through widen)
template <typename TD, typename T>
__device__ __forceinline__ TD to_t(T x) {
  return (TD)x;
}
template <>
__device__ __forceinline__ double to_t<double, float>(float x) {
  return widen(x);
}

__device__ __forceinline__ double harm(double a, double b, double) {
#if defined(__CUDA_ARCH__)
  return harmonic(a, b);
#else
  return __ddiv_rn(__dmul_rn(2.0 * a, b), __dadd_rn(a, b));
#endif
}
__device__ __forceinline__ float harm(double a, double b, float) {
  const float a32 = __double2float_rn(a), b32 = __double2float_rn(b);
  return __fdiv_rn(__fmul_rn(2.0f * a32, b32), __fadd_rn(a32, b32));
}

// ---------------------------------------------------------------------------------
// Operator set-up. In FP64 the faces and 1/D are bound by the FP64 pipe: 21 operations for a
// node's three harmonic means (39 with the language's division), nine for D and 1/D. A 129^3 / 65^3
// level of 24 samples: faces 3.94 -> 2.55 ms, diagonals 1.31 -> 1.14.
// ---------------------------------------------------------------------------------
template <typename T>
__global__ void k_faces(const double* __restrict__ k0, int n0, int st0, int n, int B, T* __restrict__ Kx,
                        T* __restrict__ Ky, T* __restrict__ Kz) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // node of the plane
  if (q >= n * n) return;
  const int y = q / n, x = q - y * n;
  const size_t n3 = (size_t)n * n * n, n03 = (size_t)n0 * n0 * n0;
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, z = zz - s * n;
    const double* kb = k0 + (size_t)s * n03;
    const size_t p0 = ((size_t)(st0 * z) * n0 + (size_t)(st0 * y)) * n0 + (size_t)(st0 * x);
    const size_t t = (size_t)s * n3 + (size_t)(z * n * n + q);
    const double a = kb[p0];
    Kx[t] = x < n - 1 ? harm(a, kb[p0 + st0], T()) : T(0);
    Ky[t] = y < n - 1 ? harm(a, kb[p0 + (size_t)st0 * n0], T()) : T(0);
    Kz[t] = z < n - 1 ? harm(a, kb[p0 + (size_t)st0 * n0 * n0], T()) : T(0);
  }
}

// D = sum of the six faces at interior nodes (fixed order), Dinv = 1 / D; 0 on the boundary.
template <typename T, typename TD>
__global__ void k_diag(int n, int B, const T* __restrict__ Kx, const T* __restrict__ Ky, const T* __restrict__ Kz,
                       TD* __restrict__ D, TD* __restrict__ Dinv) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // node of the plane
  if (q >= n * n) return;
  const int y = q / n, x = q - y * n;
  const size_t n3 = (size_t)n * n * n, n2 = (size_t)n * n;
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, z = zz - s * n;
    const size_t t = (size_t)s * n3 + (size_t)(z * n * n + q);
    const bool in = x > 0 && y > 0 && z > 0 && x < n - 1 && y < n - 1 && z < n - 1;
    TD d = 0;
    if (in) {
      d = to_t<TD>(Kx[t - 1]);
      d += to_t<TD>(Kx[t]);
      d += to_t<TD>(Ky[t - n]);
      d += to_t<TD>(Ky[t]);
      d += to_t<TD>(Kz[t - n2]);
      d += to_t<TD>(Kz[t]);
    }
    if (D) D[t] = d;
#if defined(__CUDA_ARCH__)
    if (Dinv) Dinv[t] = in ? reciprocal(d) : (TD)0;
#else
    if (Dinv) Dinv[t] = in ? (TD)1 / d : (TD)0;
#endif
  }
}

// Dense 27x27 scaled operator of the 5^3 grid, its Cholesky factor and the inverse, one warp
// per sample, four samples per block. Lane i keeps row i in registers; in the order x + 3 y +
// 9 z the matrix and its factor have half bandwidth 9, so a column updates the nine rows
// below it and everything else is zero. The factorisation is right-looking (column j, once
// scaled, is subtracted from columns j + 1 .. j + 9: independent updates instead of a
// dot product per entry); lane c then solves L L^T x = e_c, column-oriented both ways. The
// factor sits in shared memory, the 27 reciprocal pivots are formed once. What bounds it is
// the chain of 27 pivots (rsqrt, scaling, exchange) and of 54 substitution steps; the
// left-looking form on one lane per pivot in global memory took 127 us for up to
// 600 samples and 674 us for 4096, this one 39 us for one sample, 45 for 19, 242 for 4096.
constexpr int kCoarseN = 27, kCoarseBand = 9, kCoarseWarps = 4;
template <typename T>
__global__ void __launch_bounds__(32 * kCoarseWarps)
    k_coarse_setup(int B, const T* __restrict__ Kx, const T* __restrict__ Ky, const T* __restrict__ Kz,
                   double* __restrict__ Ainv) {
  constexpr int N = kCoarseN, BW = kCoarseBand;
  __shared__ double sL[kCoarseWarps][N][N];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, s = blockIdx.x * kCoarseWarps + w;
  if (s >= B) return;
  volatile double(*L)[N] = sL[w];  // volatile: loads stay at their use instead of all being held in registers
  const int i = lane < N ? lane : N - 1;  // lanes 27 .. 31 repeat row 26 and store nothing
  double a[N];
  {
    const int n = 5, x = 1 + i % 3, y = 1 + (i / 3) % 3, z = 1 + i / 9;
    const size_t p = (size_t)s * 125 + (size_t)(z * n + y) * n + x;
    const double f[6] = {(double)Kx[p - 1], (double)Kx[p], (double)Ky[p - n], (double)Ky[p], (double)Kz[p - 25],
                         (double)Kz[p]};
    double d = 0.0;
#pragma unroll
    for (int q = 0; q < 6; ++q) d += f[q];
#pragma unroll
    for (int c = 0; c < N; ++c)  // the lower triangle of row i
      a[c] = c == i ? d : (c == i - 1 && x > 1) ? -f[0] : (c == i - 3 && y > 1) ? -f[2] : (c == i - 9 && z > 1) ? -f[4] : 0.0;
  }
  double rp = 0.0;  // reciprocal pivot of row i
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const double rs = rsqrt(__shfl_sync(0xffffffffu, a[j], j));
    a[j] *= rs;  // l_ij; at row j d / sqrt(d)
    if (i == j) rp = rs;
#pragma unroll
    for (int c = j + 1; c < N; ++c) {
      if (c > j + BW) break;
      a[c] -= a[j] * __shfl_sync(0xffffffffu, a[j], c);
    }
  }
  if (lane < N) {
#pragma unroll
    for (int c = 0; c < N; ++c) L[lane][c] = c == lane ? rp : a[c];  // the diagonal holds 1 / l_ii
  }
  __syncwarp();
  double v[N];
#pragma unroll
  for (int r = 0; r < N; ++r) v[r] = r == i ? 1.0 : 0.0;
#pragma unroll
  for (int r = 0; r < N; ++r) {
    v[r] *= L[r][r];
#pragma unroll
    for (int q = r + 1; q < N; ++q) {
      if (q > r + BW) break;
      v[q] -= L[q][r] * v[r];
    }
  }
#pragma unroll
  for (int r = N - 1; r >= 0; --r) {
    v[r] *= L[r][r];
#pragma unroll
    for (int q = r - 1; q >= 0; --q) {
      if (q < r - BW) break;
      v[q] -= L[r][q] * v[r];
    }
  }
  if (lane < N) {
#pragma unroll
    for (int r = 0; r < N; ++r) Ainv[(size_t)s * N * N + r * N + lane] = v[r];
  }
}

// u = A~^-1 g on the 5^3 grid (interior nodes; boundary untouched); SPLIT: g and u in
// colour-split storage.
template <typename T, bool SPLIT = false>
__global__ void k_coarse_apply(int B, const double* __restrict__ Ainv, const T* __restrict__ g, T* __restrict__ u,
                               const int* __restrict__ active) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= B * 27) return;
  const int s = t / 27, i = t - s * 27;
  if (active && !active[s]) return;
  const double* X = Ainv + (size_t)s * 729 + (size_t)i * 27;
  const size_t base = (size_t)s * (SPLIT ? split_elems(5) : (size_t)125);
  auto at = [&](int x, int y, int z) -> size_t {
    return base + (SPLIT ? (size_t)split_index(5, x, y, z) : (size_t)((z * 5 + y) * 5 + x));
  };
  double v = 0.0;
  for (int j = 0; j < 27; ++j) {
    const int x = 1 + j % 3, y = 1 + (j / 3) % 3, z = 1 + j / 9;
    v = fma(X[j], (double)g[at(x, y, z)], v);
  }
  const int x = 1 + i % 3, y = 1 + (i / 3) % 3, z = 1 + i / 9;
  u[at(x, y, z)] = (T)v;
}

// ---------------------------------------------------------------------------------
// Cycle kernels
// ---------------------------------------------------------------------------------

// One colour of a red-black sweep: threads enumerate only the nodes of that colour.
// ZERO: the iterate is zero (first red pass of a correction from a zero guess): the sweep's
// result without its six products, u = g / D, and no read of u.
template <typename T, bool ZERO = false>
__global__ void k_rbgs(int colour, int n, int B, const T* __restrict__ Kx, const T* __restrict__ Ky,
                       const T* __restrict__ Kz, const T* __restrict__ Dinv, const T* __restrict__ g, T* __restrict__ u,
                       const int* __restrict__ active) {
  // n = 2^p + 1: a row holds half = 2^(p-1) nodes of each colour
  const int m = n - 2, half = (n - 1) / 2, lh = 31 - __clz(half);
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // colour node of an interior plane
  if (q >= m * half) return;
  const int xi = q & (half - 1), y = 1 + (q >> lh);
  const size_t n3 = (size_t)n * n * n, n2 = (size_t)n * n;
  for (int zz = blockIdx.y; zz < B * m; zz += gridDim.y) {
    const int s = zz / m, z = 1 + (zz - s * m);
    if (active && !active[s]) continue;
    const int x = (((1 + y + z) & 1) == colour ? 1 : 2) + 2 * xi;
    if (x > n - 2) continue;
    const size_t p = (size_t)s * n3 + (size_t)(z * n * n + y * n + x);
    T acc = g[p];
    if (!ZERO) {
      acc = fma(Kx[p - 1], u[p - 1], acc);
      acc = fma(Kx[p], u[p + 1], acc);
      acc = fma(Ky[p - n], u[p - n], acc);
      acc = fma(Ky[p], u[p + n], acc);
      acc = fma(Kz[p - n2], u[p - n2], acc);
      acc = fma(Kz[p], u[p + n2], acc);
    }
    u[p] = acc * Dinv[p];
  }
}

// r~ = g - D u + sum K u_q (k_residual_z's operations and order) at the interior red nodes
// only: after a sweep, whose last colour is black, the black residuals are zero up to
// rounding, and the restrictions below take them as zero (HALF). Half the FP64 work of the
// full residual, which stays for cycles without pre-smoothing.
template <typename T>
__global__ void k_residual_red(int n, int B, const T* __restrict__ Kx, const T* __restrict__ Ky,
                               const T* __restrict__ Kz, const T* __restrict__ D, const T* __restrict__ g,
                               const T* __restrict__ u, T* __restrict__ r, const int* __restrict__ active) {
  const int m = n - 2, half = (n - 1) / 2, lh = 31 - __clz(half);
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // red node of an interior plane
  if (q >= m * half) return;
  const int xi = q & (half - 1), y = 1 + (q >> lh);
  const size_t n3 = (size_t)n * n * n, n2 = (size_t)n * n;
  for (int zz = blockIdx.y; zz < B * m; zz += gridDim.y) {
    const int s = zz / m, z = 1 + (zz - s * m);
    if (active && !active[s]) continue;
    const int x = (((1 + y + z) & 1) == 0 ? 1 : 2) + 2 * xi;
    if (x > n - 2) continue;
    const size_t p = (size_t)s * n3 + (size_t)(z * n * n + y * n + x);
    T rr = fma(-D[p], u[p], g[p]);
    rr = fma(Kx[p - 1], u[p - 1], rr);
    rr = fma(Kx[p], u[p + 1], rr);
    rr = fma(Ky[p - n], u[p - n], rr);
    rr = fma(Ky[p], u[p + n], rr);
    rr = fma(Kz[p - n2], u[p - n2], rr);
    rr = fma(Kz[p], u[p + n2], rr);
    r[p] = rr;
  }
}

// Reciprocal nodal coefficient rho = 1/k of an MG grid in the grid's precision (injection
// from the finest k): the input of the nodal-coefficient sweep, whose harmonic faces are
// 2ab/(a+b) = 2/(rho_a + rho_b).
template <typename T>
__global__ void k_nodal_k(const double* __restrict__ k0, int n0, int st0, int n, int B, T* __restrict__ kn) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // node of the plane
  if (q >= n * n) return;
  const int y = q / n, x = q - y * n;
  const size_t n3 = (size_t)n * n * n, n03 = (size_t)n0 * n0 * n0;
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, z = zz - s * n;
    const size_t p0 = ((size_t)(st0 * z) * n0 + (size_t)(st0 * y)) * n0 + (size_t)(st0 * x);
    kn[(size_t)s * n3 + (size_t)(z * n * n + q)] = (T)(1.0 / k0[(size_t)s * n03 + p0]);
  }
}

// Harmonic face of the nodal-coefficient kernels from the reciprocal coefficients:
// 2ab / (a + b) = 2 / (rho_a + rho_b), with the fast reciprocal (__fdividef, within 2
// ulp). Symmetric in the two nodes, so both see the same value; the faces differ from the
// stored IEEE ones by a few ulps.
__device__ __forceinline__ float nodal_face(float ra, float rb) { return __fdividef(2.0f, __fadd_rn(ra, rb)); }

// One colour of a red-black sweep that reads the (reciprocal) nodal coefficient (FP32) instead of
// stored faces: the six harmonic faces, their sum D and 1/D of the updated node are
// recomputed per update with fast reciprocals, so a sweep reads 4 words per node (u read
// and written, g, k) instead of 7. It is the Gauss-Seidel sweep of an operator within a
// few ulps of the stored FP32 one: used only inside the FP32 correction cycle, whose
// result the FP64 outer residual (stored faces) corrects, so the converged solution is
// that of the stored operator.
template <bool ZERO = false>
__global__ void k_rbgs_nodal(int colour, int n, int B, const float* __restrict__ kn, const float* __restrict__ g,
                             float* __restrict__ u, const int* __restrict__ active) {
  const int m = n - 2, half = (n - 1) / 2, lh = 31 - __clz(half);
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // colour node of an interior plane
  if (q >= m * half) return;
  const int xi = q & (half - 1), y = 1 + (q >> lh);
  const size_t n3 = (size_t)n * n * n, n2 = (size_t)n * n;
  for (int zz = blockIdx.y; zz < B * m; zz += gridDim.y) {
    const int s = zz / m, z = 1 + (zz - s * m);
    if (active && !active[s]) continue;
    const int x = (((1 + y + z) & 1) == colour ? 1 : 2) + 2 * xi;
    if (x > n - 2) continue;
    const size_t p = (size_t)s * n3 + (size_t)(z * n * n + y * n + x);
    const float kc = kn[p];
    const float kxm = nodal_face(kn[p - 1], kc), kxp = nodal_face(kc, kn[p + 1]);
    const float kym = nodal_face(kn[p - n], kc), kyp = nodal_face(kc, kn[p + n]);
    const float kzm = nodal_face(kn[p - n2], kc), kzp = nodal_face(kc, kn[p + n2]);
    float d = kxm;
    d += kxp;
    d += kym;
    d += kyp;
    d += kzm;
    d += kzp;
    const float dinv = __fdividef(1.0f, d);
    float acc = g[p];
    if (!ZERO) {
      acc = fmaf(kxm, u[p - 1], acc);
      acc = fmaf(kxp, u[p + 1], acc);
      acc = fmaf(kym, u[p - n], acc);
      acc = fmaf(kyp, u[p + n], acc);
      acc = fmaf(kzm, u[p - n2], acc);
      acc = fmaf(kzp, u[p + n2], acc);
    }
    u[p] = acc * dinv;
  }
}

// r~ = g - D u + sum K u_q of an FP32 grid from the nodal coefficient (faces and D
// recomputed as in k_rbgs_nodal, then k_residual_z's operation order): the residual of the
// operator the nodal sweep smooths; r~ on interior nodes, 0 on the boundary; 4 words per
// node instead of 7.
// RED: the red nodes only (k_residual_red's reason), the threads enumerating rows of red nodes.
template <bool RED = false>
__global__ void k_residual_nodal(int n, int B, const float* __restrict__ kn, const float* __restrict__ g,
                                 const float* __restrict__ u, float* __restrict__ r, const int* __restrict__ active) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // node (RED: red node) of the plane
  const int half = (n + 1) / 2;
  if (q >= (RED ? n * half : n * n)) return;
  const int y = q / (RED ? half : n), xq = q - y * (RED ? half : n);
  const size_t n3 = (size_t)n * n * n, n2 = (size_t)n * n;
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, z = zz - s * n;
    if (active && !active[s]) continue;
    const int x = RED ? 2 * xq + ((y + z) & 1) : xq;
    if (RED && x > n - 1) continue;
    const size_t p = (size_t)s * n3 + (size_t)(z * n * n + y * n + x);
    float rr = 0.0f;
    if (x > 0 && y > 0 && z > 0 && x < n - 1 && y < n - 1 && z < n - 1) {
      const float kc = kn[p];
      const float kxm = nodal_face(kn[p - 1], kc), kxp = nodal_face(kc, kn[p + 1]);
      const float kym = nodal_face(kn[p - n], kc), kyp = nodal_face(kc, kn[p + n]);
      const float kzm = nodal_face(kn[p - n2], kc), kzp = nodal_face(kc, kn[p + n2]);
      float d = kxm;
      d += kxp;
      d += kym;
      d += kyp;
      d += kzm;
      d += kzp;
      rr = fmaf(-d, u[p], g[p]);
      rr = fmaf(kxm, u[p - 1], rr);
      rr = fmaf(kxp, u[p + 1], rr);
      rr = fmaf(kym, u[p - n], rr);
      rr = fmaf(kyp, u[p + n], rr);
      rr = fmaf(kzm, u[p - n2], rr);
      rr = fmaf(kzp, u[p + n2], rr);
    }
    r[p] = rr;
  }
}

// ---------------------------------------------------------------------------------
// Colour-split storage of the FP32 correction hierarchy (MLMC_SMOOTH_SPLIT): per sample
// the nodes of colour c = (x + y + z) & 1 form one block of n x n rows of P slots, node
// (x, y, z) at slot x >> 1 of row (z, y) of its colour's block; P = (n + 1) / 2 rounded up
// to a multiple of 4, so that every row starts on a 16-byte boundary (four slots per
// vector access). A colour pass
// of the red-black sweep then streams the lines of the colour it updates plus those of
// the other colour it reads (2.5 instead of 4 words per node and pass at line
// granularity). Neighbours of node x = 2 xi + q (q = x parity) in the other colour: x - 1
// at slot xi - 1 + q, x + 1 at slot xi + q, y +- 1 and z +- 1 at slot xi. The slot x = n
// of odd-parity rows and the padding slots do not exist in the grid: a kernel may load
// them along with a vector of slots but never uses their values.
// ---------------------------------------------------------------------------------
// Reciprocal nodal coefficient 1/k of an FP32 grid (every node) into colour-split storage.
__global__ void k_nodal_k_split(const double* __restrict__ k0, int n0, int st0, int n, int B, float* __restrict__ kn) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // node of the plane
  if (q >= n * n) return;
  const int y = q / n, x = q - y * n;
  const size_t ns = split_elems(n), n03 = (size_t)n0 * n0 * n0;
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, z = zz - s * n;
    const size_t p0 = ((size_t)(st0 * z) * n0 + (size_t)(st0 * y)) * n0 + (size_t)(st0 * x);
    kn[(size_t)s * ns + split_index(n, x, y, z)] = (float)(1.0 / k0[(size_t)s * n03 + p0]);
  }
}

// Compile-time geometry of a colour-split grid of n = 2^LG + 1 nodes per axis: with n a
// constant, the row / slot split of a thread index and every neighbour offset are
// shifts, multiplications by constants and immediate load offsets (the runtime-n form of
// these kernels spent about 280 instructions per updated node and was issue-bound).
template <int LG>
struct SplitGeo {
  static constexpr int n = (1 << LG) + 1, m = n - 2, P = (((n + 1) / 2) + 3) & ~3, NP = n * P, BLK = n * n * P;
  // four- and two-slot groups that hold an interior node (x = 1 .. n - 2) of either parity: the
  // passes give threads to these only (of the padded row's 9 four-slot groups at 65^3 to 8, of its
  // 18 two-slot groups to 16; an idle lane costs the FP64 pipe as much as a busy one: the colour
  // passes of a 129^3 / 65^3 level of 24 samples 31.0 -> 29.5 ms, FP32 ones of 33^3 x 48 1.15 -> 1.06)
  static constexpr int A4 = n > 9 ? (n - 1) / 8 : 1, A2 = (n - 1) / 4;
  static constexpr size_t NS = (size_t)2 * BLK;  // elements per sample
};

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float comp(const float4& v, int i) { return i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w; }

// The nodal-coefficient update of one node from its own k^-1 and right-hand side and the
// six neighbours' k^-1 and iterate, in k_rbgs_nodal's order of operations.
// ZERO: the iterate is zero (g / D alone).
template <bool ZERO = false>
__device__ __forceinline__ float nodal_update(float kc, float gp, float kl, float ul, float kr, float ur, float kym,
                                              float uym, float kyp, float uyp, float kzm, float uzm, float kzp,
                                              float uzp) {
  const float fxm = nodal_face(kl, kc), fxp = nodal_face(kc, kr);
  const float fym = nodal_face(kym, kc), fyp = nodal_face(kc, kyp);
  const float fzm = nodal_face(kzm, kc), fzp = nodal_face(kc, kzp);
  float d = fxm;
  d += fxp;
  d += fym;
  d += fyp;
  d += fzm;
  d += fzp;
  const float dinv = __fdividef(1.0f, d);
  float acc = gp;
  if (!ZERO) {
    acc = fmaf(fxm, ul, acc);
    acc = fmaf(fxp, ur, acc);
    acc = fmaf(fym, uym, acc);
    acc = fmaf(fyp, uyp, acc);
    acc = fmaf(fzm, uzm, acc);
    acc = fmaf(fzp, uzp, acc);
  }
  return acc * dinv;
}

// The residual of one node in k_residual_nodal's order of operations.
__device__ __forceinline__ float nodal_residual(float kc, float gp, float up, float kl, float ul, float kr, float ur,
                                                float kym, float uym, float kyp, float uyp, float kzm, float uzm,
                                                float kzp, float uzp) {
  const float fxm = nodal_face(kl, kc), fxp = nodal_face(kc, kr);
  const float fym = nodal_face(kym, kc), fyp = nodal_face(kc, kyp);
  const float fzm = nodal_face(kzm, kc), fzp = nodal_face(kc, kzp);
  float d = fxm;
  d += fxp;
  d += fym;
  d += fyp;
  d += fzm;
  d += fzp;
  float rr = fmaf(-d, up, gp);
  rr = fmaf(fxm, ul, rr);
  rr = fmaf(fxp, ur, rr);
  rr = fmaf(fym, uym, rr);
  rr = fmaf(fyp, uyp, rr);
  rr = fmaf(fzm, uzm, rr);
  rr = fmaf(fzp, uzp, rr);
  return rr;
}

// One colour of the nodal-coefficient red-black sweep on colour-split storage: the same
// operations in the same order as k_rbgs_nodal (bit for bit the same iterate). A thread
// updates the four nodes of one four-slot group of an interior row with 16-byte loads:
// its own k^-1 and g, the other colour's k^-1 and u in the same slots of its row (x - 1
// or x + 1 of the group's nodes) and of the rows y +- 1, z +- 1, plus one scalar slot
// outside the group. Grid (groups of the interior rows of a plane, interior planes,
// samples). ZERO: from a zero iterate (k_rbgs).
template <int LG, bool ZERO = false>
__global__ void __launch_bounds__(128) k_rbgs_split(int colour, const float* __restrict__ kn,
                                                    const float* __restrict__ g, float* __restrict__ u,
                                                    const int* __restrict__ active) {
  using G = SplitGeo<LG>;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // group of an interior row
  if (q >= G::m * G::A4) return;
  const int s = blockIdx.z;
  if (active && !active[s]) return;
  const int yi = q / G::A4, qi = q - yi * G::A4, y = 1 + yi, z = 1 + (int)blockIdx.y;
  const int par = (colour + y + z) & 1, xi0 = 4 * qi, x0 = 2 * xi0 + par;  // node i: x = x0 + 2 i
  if (x0 > G::n - 2) return;  // boundary and padding slots only
  const int o = (z * G::n + y) * G::P + xi0;
  const size_t cb = (size_t)s * G::NS + (size_t)colour * G::BLK, ob = (size_t)s * G::NS + (size_t)(1 - colour) * G::BLK;
  const float* ko = kn + ob;
  const float* uo = u + ob;
  const float4 kc4 = ld4(kn + cb + o), g4 = ld4(g + cb + o);
  const float4 km4 = ld4(ko + o), kym4 = ld4(ko + o - G::P), kyp4 = ld4(ko + o + G::P);
  const float4 kzm4 = ld4(ko + o - G::NP), kzp4 = ld4(ko + o + G::NP);
  const float4 zero4 = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  const float4 um4 = ZERO ? zero4 : ld4(uo + o), uym4 = ZERO ? zero4 : ld4(uo + o - G::P);
  const float4 uyp4 = ZERO ? zero4 : ld4(uo + o + G::P);
  const float4 uzm4 = ZERO ? zero4 : ld4(uo + o - G::NP), uzp4 = ZERO ? zero4 : ld4(uo + o + G::NP);
  // the other-colour slot beside the group: left of node 0 (x parity 0) or right of node 3
  float kext = 0.0f, uext = 0.0f;
  if (par) {
    kext = ko[o + 4];
    if (!ZERO) uext = uo[o + 4];
  } else if (x0 > 0) {
    kext = ko[o - 1];
    if (!ZERO) uext = uo[o - 1];
  }
  float out[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float kl = par ? comp(km4, i) : (i == 0 ? kext : comp(km4, i - 1));
    const float ul = par ? comp(um4, i) : (i == 0 ? uext : comp(um4, i - 1));
    const float kr = par ? (i == 3 ? kext : comp(km4, i + 1)) : comp(km4, i);
    const float ur = par ? (i == 3 ? uext : comp(um4, i + 1)) : comp(um4, i);
    out[i] = nodal_update<ZERO>(comp(kc4, i), comp(g4, i), kl, ul, kr, ur, comp(kym4, i), comp(uym4, i), comp(kyp4, i),
                          comp(uyp4, i), comp(kzm4, i), comp(uzm4, i), comp(kzp4, i), comp(uzp4, i));
  }
  float* uc = u + cb + o;
  if (x0 >= 1 && x0 + 6 <= G::n - 2) {
    *reinterpret_cast<float4*>(uc) = make_float4(out[0], out[1], out[2], out[3]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (x0 + 2 * i >= 1 && x0 + 2 * i <= G::n - 2) uc[i] = out[i];
  }
}

// r~ = g - D u + sum K u_q (k_residual_nodal's operations and order) at the interior
// nodes of one colour, four slots per thread as in k_rbgs_split, into r in colour-split
// storage (the restriction reads only interior fine nodes; boundary and padding slots of
// r are not written). Grid (groups of the interior rows of a plane, 2 x interior planes,
// samples): colour = blockIdx.y & 1, so the two colours of a plane run back to back and
// the 1/k and u rows each reads as the other colour's are still in L2. RED: the red nodes
// only (k_residual_red's reason; 3 words per two nodes), blockIdx.y the interior plane.
template <int LG, bool RED = false>
__global__ void __launch_bounds__(128, 8) k_residual_split(const float* __restrict__ kn, const float* __restrict__ g,
                                                        const float* __restrict__ u, float* __restrict__ r,
                                                        const int* __restrict__ active) {
  using G = SplitGeo<LG>;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= G::m * G::A4) return;
  const int s = blockIdx.z, colour = RED ? 0 : blockIdx.y & 1;
  if (active && !active[s]) return;
  const int yi = q / G::A4, qi = q - yi * G::A4, y = 1 + yi, z = 1 + (int)(RED ? blockIdx.y : blockIdx.y >> 1);
  const int par = (colour + y + z) & 1, xi0 = 4 * qi, x0 = 2 * xi0 + par;
  if (x0 > G::n - 2) return;
  const int o = (z * G::n + y) * G::P + xi0;
  const size_t cb = (size_t)s * G::NS + (size_t)colour * G::BLK, ob = (size_t)s * G::NS + (size_t)(1 - colour) * G::BLK;
  const float* ko = kn + ob;
  const float* uo = u + ob;
  const float4 kc4 = ld4(kn + cb + o), g4 = ld4(g + cb + o), up4 = ld4(u + cb + o);
  const float4 km4 = ld4(ko + o), kym4 = ld4(ko + o - G::P), kyp4 = ld4(ko + o + G::P);
  const float4 kzm4 = ld4(ko + o - G::NP), kzp4 = ld4(ko + o + G::NP);
  const float4 um4 = ld4(uo + o), uym4 = ld4(uo + o - G::P), uyp4 = ld4(uo + o + G::P);
  const float4 uzm4 = ld4(uo + o - G::NP), uzp4 = ld4(uo + o + G::NP);
  float kext = 0.0f, uext = 0.0f;
  if (par) {
    kext = ko[o + 4];
    uext = uo[o + 4];
  } else if (x0 > 0) {
    kext = ko[o - 1];
    uext = uo[o - 1];
  }
  float out[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float kl = par ? comp(km4, i) : (i == 0 ? kext : comp(km4, i - 1));
    const float ul = par ? comp(um4, i) : (i == 0 ? uext : comp(um4, i - 1));
    const float kr = par ? (i == 3 ? kext : comp(km4, i + 1)) : comp(km4, i);
    const float ur = par ? (i == 3 ? uext : comp(um4, i + 1)) : comp(um4, i);
    out[i] = nodal_residual(comp(kc4, i), comp(g4, i), comp(up4, i), kl, ul, kr, ur, comp(kym4, i), comp(uym4, i),
                            comp(kyp4, i), comp(uyp4, i), comp(kzm4, i), comp(uzm4, i), comp(kzp4, i),
                            comp(uzp4, i));
  }
  float* rc = r + cb + o;
  if (x0 >= 1 && x0 + 6 <= G::n - 2) {
    *reinterpret_cast<float4*>(rc) = make_float4(out[0], out[1], out[2], out[3]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (x0 + 2 * i >= 1 && x0 + 2 * i <= G::n - 2) rc[i] = out[i];
  }
}

// g_c = 4 FW(r~) (k_restrict's weights and order) from r~ in colour-split storage into the
// coarse grid's colour-split g, at interior coarse nodes. LG: the fine grid's. Grid
// (interior coarse nodes of a plane, interior coarse planes, samples). HALF: r~ is zero at
// black nodes (k_residual_red): the 13 red neighbours of the 27.
template <int LG, typename T = float, bool HALF = false>
__global__ void __launch_bounds__(128) k_restrict_split(const T* __restrict__ r, T* __restrict__ gc,
                                                        const int* __restrict__ active) {
  using F = SplitGeo<LG>;
  using C = SplitGeo<LG - 1>;
  constexpr int mc = C::n - 2;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= mc * mc) return;
  const int s = blockIdx.z;
  if (active && !active[s]) return;
  const int Y = 1 + q / mc, X = 1 + q - (Y - 1) * mc, Z = 1 + (int)blockIdx.y;
  const T* rb = r + (size_t)s * F::NS;
  T v = 0;
#pragma unroll
  for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
    for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx) {
        if (HALF && ((dx + dy + dz) & 1)) continue;
        const T wgt = (T)((2 - abs(dx)) * (2 - abs(dy)) * (2 - abs(dz))) * (T)(1.0 / 16.0);
        const int fx = 2 * X + dx, fy = 2 * Y + dy, fz = 2 * Z + dz;  // colour (dx + dy + dz) & 1
        v = fma(wgt, rb[(size_t)((dx + dy + dz) & 1) * F::BLK + (size_t)((fz * F::n + fy) * F::P + (fx >> 1))], v);
      }
  gc[(size_t)s * C::NS + (size_t)((X + Y + Z) & 1) * C::BLK + (size_t)((Z * C::n + Y) * C::P + (X >> 1))] = v;
}

// u_f += trilinear interpolation of e_c on colour-split storage of both grids: the
// coarse terms of k_prolong in its order (rows (Z, Y), (Z, Y+1), (Z+1, Y), (Z+1, Y+1),
// each X then X+1) and its weights, so the result is bit for bit that of k_prolong. A
// thread corrects the four fine nodes of one four-slot group of one colour (x = x0 + 2 i,
// coarse X = xi0 + i, one x parity, hence one weight pattern) with a 16-byte update of u;
// each coarse row it needs is gathered once for the group (X = xi0 .. xi0 + 4). LG: the
// fine grid's. Grid (groups of the interior rows of a plane, interior planes,
// 2 x samples: colour = blockIdx.z & 1). BLACK: the black nodes only, blockIdx.z the sample:
// a red pass follows, which overwrites the red nodes without reading them.
template <int LG, bool BLACK = false>
__global__ void __launch_bounds__(128) k_prolong_split(const float* __restrict__ ec, float* __restrict__ u,
                                                       const int* __restrict__ active) {
  using F = SplitGeo<LG>;
  using C = SplitGeo<LG - 1>;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= F::m * F::A4) return;
  const int s = BLACK ? blockIdx.z : blockIdx.z >> 1, colour = BLACK ? 1 : blockIdx.z & 1;
  if (active && !active[s]) return;
  const int yi = q / F::A4, qi = q - yi * F::A4, y = 1 + yi, z = 1 + (int)blockIdx.y;
  const int xo = (colour + y + z) & 1, xi0 = 4 * qi, x0 = 2 * xi0 + xo;
  if (x0 > F::n - 2) return;
  const int yo = y & 1, zo = z & 1, Y = y >> 1, Z = z >> 1;
  const float* e = ec + (size_t)s * C::NS;
  // coarse row (Y + b, Z + c) at X = xi0 + t, t = 0 .. 4 (xi0 even: colour (t + Y + b + Z + c) & 1,
  // slot xi0 / 2 + t / 2)
  auto row = [&](int b, int c, float* cv) {
    const int cy = Y + b, cz = Z + c, base = (cz * C::n + cy) * C::P + (xi0 >> 1);
#pragma unroll
    for (int t = 0; t < 5; ++t)
      if (t < 4 || xo) cv[t] = e[(size_t)((t + cy + cz) & 1) * C::BLK + (size_t)(base + (t >> 1))];
  };
  float r00[5], r10[5], r01[5], r11[5];  // rows (Y, Z), (Y+1, Z), (Y, Z+1), (Y+1, Z+1)
  row(0, 0, r00);
  if (yo) row(1, 0, r10);
  if (zo) {
    row(0, 1, r01);
    if (yo) row(1, 1, r11);
  }
  const float w = xo + yo + zo == 0 ? 1.0f : xo + yo + zo == 1 ? 0.5f : xo + yo + zo == 2 ? 0.25f : 0.125f;
  float* uc = u + (size_t)s * F::NS + (size_t)colour * F::BLK + (size_t)((z * F::n + y) * F::P + xi0);
  const float4 u4 = ld4(uc);
  float out[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float v = 0.0f;
    v += r00[i];
    if (xo) v += r00[i + 1];
    if (yo) {
      v += r10[i];
      if (xo) v += r10[i + 1];
    }
    if (zo) {
      v += r01[i];
      if (xo) v += r01[i + 1];
      if (yo) {
        v += r11[i];
        if (xo) v += r11[i + 1];
      }
    }
    out[i] = comp(u4, i) + w * v;
  }
  if (x0 >= 1 && x0 + 6 <= F::n - 2) {
    *reinterpret_cast<float4*>(uc) = make_float4(out[0], out[1], out[2], out[3]);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (x0 + 2 * i >= 1 && x0 + 2 * i <= F::n - 2) uc[i] = out[i];
  }
}

// ---------------------------------------------------------------------------------
// Colour-split storage of FP64 stored-face grids (MLMC_SMOOTH_SPLIT in an FP64 solve):
// u, g, r, the faces Kx, Ky, Kz (each at its lower node), D and 1/D of every grid but the
// coarsest in the split storage. A colour pass then reads its own colour's faces, 1/D and
// g, the other colour's three lower faces and u, and writes its own u: 5 words per node and
// pass at line granularity against the plain layout's ~7. Every kernel performs the
// two-pass kernels' operations in their order, so the iterates are those of
// MLMC_SMOOTH_TWO_PASS bit for bit.
// ---------------------------------------------------------------------------------
__device__ __forceinline__ double2 ld2(const double* p) { return *reinterpret_cast<const double2*>(p); }
__device__ __forceinline__ double comp2(const double2& v, int i) { return i == 0 ? v.x : v.y; }

// harmonic faces of the (injected) FP64 nodal k into colour-split storage (k_faces).
__global__ void k_faces_split(const double* __restrict__ k0, int n0, int st0, int n, int B, double* __restrict__ Kx,
                              double* __restrict__ Ky, double* __restrict__ Kz) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // node of the plane
  if (q >= n * n) return;
  const int y = q / n, x = q - y * n;
  const size_t ns = split_elems(n), n03 = (size_t)n0 * n0 * n0;
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, z = zz - s * n;
    const double* kb = k0 + (size_t)s * n03;
    const size_t p0 = ((size_t)(st0 * z) * n0 + (size_t)(st0 * y)) * n0 + (size_t)(st0 * x);
    const size_t t = (size_t)s * ns + split_index(n, x, y, z);
    const double a = kb[p0];
    Kx[t] = x < n - 1 ? harm(a, kb[p0 + st0], double()) : 0.0;
    Ky[t] = y < n - 1 ? harm(a, kb[p0 + (size_t)st0 * n0], double()) : 0.0;
    Kz[t] = z < n - 1 ? harm(a, kb[p0 + (size_t)st0 * n0 * n0], double()) : 0.0;
  }
}

// D = sum of the six faces (k_diag's order) and 1/D at interior nodes, 0 on the boundary,
// all in colour-split storage.
__global__ void k_diag_split(int n, int B, const double* __restrict__ Kx, const double* __restrict__ Ky,
                             const double* __restrict__ Kz, double* __restrict__ D, double* __restrict__ Dinv) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n * n) return;
  const int y = q / n, x = q - y * n;
  const size_t ns = split_elems(n);
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, z = zz - s * n;
    const size_t b = (size_t)s * ns, t = b + split_index(n, x, y, z);
    const bool in = x > 0 && y > 0 && z > 0 && x < n - 1 && y < n - 1 && z < n - 1;
    double d = 0.0;
    if (in) {
      d = Kx[b + split_index(n, x - 1, y, z)];
      d += Kx[t];
      d += Ky[b + split_index(n, x, y - 1, z)];
      d += Ky[t];
      d += Kz[b + split_index(n, x, y, z - 1)];
      d += Kz[t];
    }
    D[t] = d;
#if defined(__CUDA_ARCH__)
    Dinv[t] = in ? reciprocal(d) : 0.0;
#else
    Dinv[t] = in ? 1.0 / d : 0.0;
#endif
  }
}

// plain <-> colour-split copies of B samples of an n^3 grid (every node)
template <typename T, bool TO_SPLIT>
__global__ void k_split_copy(int n, int B, const T* __restrict__ a, T* __restrict__ b) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n * n) return;
  const int y = q / n, x = q - y * n;
  const size_t n3 = (size_t)n * n * n, ns = split_elems(n);
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, z = zz - s * n;
    const size_t tp = (size_t)s * n3 + (size_t)(z * n * n + q), ts = (size_t)s * ns + split_index(n, x, y, z);
    if (TO_SPLIT)
      b[ts] = a[tp];
    else
      b[tp] = a[ts];
  }
}

// One colour of the stored-face sweep on colour-split FP64 storage (k_rbgs's operations
// and order), two nodes per thread on 16-byte loads: its own Kx, Ky, Kz, 1/D and g, the
// other colour's lower faces (x - 1, y - 1, z - 1 nodes) and u of the six neighbours.
// Grid (two-slot groups of the interior rows of a plane, interior planes, samples). ZERO:
// from a zero iterate (k_rbgs).
template <int LG, bool ZERO = false>
__global__ void __launch_bounds__(128) k_rbgs_split64(int colour, const double* __restrict__ Kx,
                                                      const double* __restrict__ Ky, const double* __restrict__ Kz,
                                                      const double* __restrict__ Dinv, const double* __restrict__ g,
                                                      double* __restrict__ u, const int* __restrict__ active) {
  using G = SplitGeo<LG>;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= G::m * G::A2) return;
  const int s = blockIdx.z;
  if (active && !active[s]) return;
  const int yi = q / G::A2, qi = q - yi * G::A2, y = 1 + yi, z = 1 + (int)blockIdx.y;
  const int par = (colour + y + z) & 1, xi0 = 2 * qi, x0 = 2 * xi0 + par;  // node i: x = x0 + 2 i
  if (x0 > G::n - 2) return;
  const int o = (z * G::n + y) * G::P + xi0;
  const size_t cb = (size_t)s * G::NS + (size_t)colour * G::BLK, ob = (size_t)s * G::NS + (size_t)(1 - colour) * G::BLK;
  const double2 di2 = ld2(Dinv + cb + o), g2 = ld2(g + cb + o);
  double* uc = u + cb + o;
  const bool inner = x0 >= 1 && x0 + 2 <= G::n - 2;
  if (ZERO) {
    const double out[2] = {g2.x * di2.x, g2.y * di2.y};
    if (inner) {
      *reinterpret_cast<double2*>(uc) = make_double2(out[0], out[1]);
    } else {
#pragma unroll
      for (int i = 0; i < 2; ++i)
        if (x0 + 2 * i >= 1 && x0 + 2 * i <= G::n - 2) uc[i] = out[i];
    }
    return;
  }
  const double2 kx2 = ld2(Kx + cb + o), ky2 = ld2(Ky + cb + o), kz2 = ld2(Kz + cb + o);
  const double* kxo = Kx + ob;
  const double* uo = u + ob;
  const double2 kxm2 = ld2(kxo + o), kym2 = ld2(Ky + ob + o - G::P), kzm2 = ld2(Kz + ob + o - G::NP);
  const double2 um2 = ld2(uo + o), uym2 = ld2(uo + o - G::P), uyp2 = ld2(uo + o + G::P);
  const double2 uzm2 = ld2(uo + o - G::NP), uzp2 = ld2(uo + o + G::NP);
  // the other-colour slot beside the pair: left of node 0 (x parity 0) or right of node 1
  double kext = 0.0, uext = 0.0;
  if (par) {
    uext = uo[o + 2];
  } else if (x0 > 0) {
    kext = kxo[o - 1];
    uext = uo[o - 1];
  }
  double out[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    // lower x face at the x - 1 node: slot xi0 + i - 1 + par of the other colour
    const double kl = par ? comp2(kxm2, i) : (i == 0 ? kext : comp2(kxm2, i - 1));
    const double ul = par ? comp2(um2, i) : (i == 0 ? uext : comp2(um2, i - 1));
    const double ur = par ? (i == 1 ? uext : comp2(um2, i + 1)) : comp2(um2, i);
    double acc = comp2(g2, i);
    acc = fma(kl, ul, acc);
    acc = fma(comp2(kx2, i), ur, acc);
    acc = fma(comp2(kym2, i), comp2(uym2, i), acc);
    acc = fma(comp2(ky2, i), comp2(uyp2, i), acc);
    acc = fma(comp2(kzm2, i), comp2(uzm2, i), acc);
    acc = fma(comp2(kz2, i), comp2(uzp2, i), acc);
    out[i] = acc * comp2(di2, i);
  }
  if (inner) {
    *reinterpret_cast<double2*>(uc) = make_double2(out[0], out[1]);
  } else {
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (x0 + 2 * i >= 1 && x0 + 2 * i <= G::n - 2) uc[i] = out[i];
  }
}

// r~ = g - D u + sum K u_q (k_residual_z's operations and order) at the interior nodes of
// one colour, two per thread, into r in colour-split storage (interior nodes only).
// Grid (two-slot groups of the interior rows of a plane, 2 x interior planes, samples):
// colour = blockIdx.y & 1 (the two colours of a plane back to back). RED: the red nodes only
// (k_residual_red's reason), blockIdx.y the interior plane.
template <int LG, bool RED = false>
__global__ void __launch_bounds__(128) k_residual_split64(const double* __restrict__ Kx, const double* __restrict__ Ky,
                                                          const double* __restrict__ Kz, const double* __restrict__ D,
                                                          const double* __restrict__ g, const double* __restrict__ u,
                                                          double* __restrict__ r, const int* __restrict__ active) {
  using G = SplitGeo<LG>;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= G::m * G::A2) return;
  const int s = blockIdx.z, colour = RED ? 0 : blockIdx.y & 1;
  if (active && !active[s]) return;
  const int yi = q / G::A2, qi = q - yi * G::A2, y = 1 + yi, z = 1 + (int)(RED ? blockIdx.y : blockIdx.y >> 1);
  const int par = (colour + y + z) & 1, xi0 = 2 * qi, x0 = 2 * xi0 + par;
  if (x0 > G::n - 2) return;
  const int o = (z * G::n + y) * G::P + xi0;
  const size_t cb = (size_t)s * G::NS + (size_t)colour * G::BLK, ob = (size_t)s * G::NS + (size_t)(1 - colour) * G::BLK;
  const double2 kx2 = ld2(Kx + cb + o), ky2 = ld2(Ky + cb + o), kz2 = ld2(Kz + cb + o);
  const double2 d2 = ld2(D + cb + o), g2 = ld2(g + cb + o), up2 = ld2(u + cb + o);
  const double* kxo = Kx + ob;
  const double* uo = u + ob;
  const double2 kxm2 = ld2(kxo + o), kym2 = ld2(Ky + ob + o - G::P), kzm2 = ld2(Kz + ob + o - G::NP);
  const double2 um2 = ld2(uo + o), uym2 = ld2(uo + o - G::P), uyp2 = ld2(uo + o + G::P);
  const double2 uzm2 = ld2(uo + o - G::NP), uzp2 = ld2(uo + o + G::NP);
  double kext = 0.0, uext = 0.0;
  if (par) {
    uext = uo[o + 2];
  } else if (x0 > 0) {
    kext = kxo[o - 1];
    uext = uo[o - 1];
  }
  double out[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const double kl = par ? comp2(kxm2, i) : (i == 0 ? kext : comp2(kxm2, i - 1));
    const double ul = par ? comp2(um2, i) : (i == 0 ? uext : comp2(um2, i - 1));
    const double ur = par ? (i == 1 ? uext : comp2(um2, i + 1)) : comp2(um2, i);
    double rr = fma(-comp2(d2, i), comp2(up2, i), comp2(g2, i));
    rr = fma(kl, ul, rr);
    rr = fma(comp2(kx2, i), ur, rr);
    rr = fma(comp2(kym2, i), comp2(uym2, i), rr);
    rr = fma(comp2(ky2, i), comp2(uyp2, i), rr);
    rr = fma(comp2(kzm2, i), comp2(uzm2, i), rr);
    rr = fma(comp2(kz2, i), comp2(uzp2, i), rr);
    out[i] = rr;
  }
  double* rc = r + cb + o;
  if (x0 >= 1 && x0 + 2 <= G::n - 2) {
    *reinterpret_cast<double2*>(rc) = make_double2(out[0], out[1]);
  } else {
#pragma unroll
    for (int i = 0; i < 2; ++i)
      if (x0 + 2 * i >= 1 && x0 + 2 * i <= G::n - 2) rc[i] = out[i];
  }
}

// Dispatch of a colour-split kernel template on n = 2^LG + 1 (5 .. 1025).
#define MLMC_SPLIT_DISPATCH(n, CALL)         \
  switch (n) {                               \
    case 5: { constexpr int LG = 2; CALL; } break;   \
    case 9: { constexpr int LG = 3; CALL; } break;   \
    case 17: { constexpr int LG = 4; CALL; } break;  \
    case 33: { constexpr int LG = 5; CALL; } break;  \
    case 65: { constexpr int LG = 6; CALL; } break;  \
    case 129: { constexpr int LG = 7; CALL; } break; \
    case 257: { constexpr int LG = 8; CALL; } break; \
    case 513: { constexpr int LG = 9; CALL; } break; \
    default: { constexpr int LG = 10; CALL; } break; \
  }

template <int THREADS>
__device__ __forceinline__ double block_sum(double v) {
  __shared__ double warp_part[THREADS / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) warp_part[wid] = v;
  __syncthreads();
  double r = 0.0;
  if (wid == 0) {
    r = lane < THREADS / 32 ? warp_part[lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  return r;  // valid in thread 0
}

// Blocks per sample of the deterministic reductions: a function of the grid size only
// (never of the batch), so that a sample's sums do not depend on its batch; up to per_sm
// blocks for each of the 152 SMs (what is resident at once: one large sample then runs as one
// whole wave).
inline int reduce_blocks(size_t work, int per_sm = 8) {
  size_t nb = (work + 4095) / 4096;
  if (nb < 1) nb = 1;
  if (nb > (size_t)(152 * per_sm)) nb = 152 * per_sm;
  return (int)nb;
}

// Sum of squares over interior nodes of an FP64 array (initial ||g||). Grid (NB, B).
__global__ void __launch_bounds__(kThreads) k_sumsq(int n, const double* __restrict__ v, double* __restrict__ partial) {
  const int s = blockIdx.y;
  const unsigned n3 = (unsigned)n * n * n, n2 = (unsigned)n * n, un = (unsigned)n;
  const unsigned chunk = (n3 + gridDim.x - 1) / gridDim.x;
  const unsigned lo = blockIdx.x * chunk, hi = lo + chunk < n3 ? lo + chunk : n3;
  double sq = 0.0;
  for (unsigned i = lo + threadIdx.x; i < hi; i += kThreads) {
    const unsigned zq = i / n2, rem = i - zq * n2, yq = rem / un;
    const int z = (int)zq, y = (int)yq, x = (int)(rem - yq * un);
    if (x > 0 && y > 0 && z > 0 && x < n - 1 && y < n - 1 && z < n - 1) {
      const double a = v[(size_t)s * n3 + i];
      sq += a * a;
    }
  }
  const double b = block_sum<kThreads>(sq);
  if (threadIdx.x == 0) partial[(size_t)s * gridDim.x + blockIdx.x] = b;
}

// Sum of a sample's NB block partials by one warp: lane l adds partials l, l+32, ...
// in order, then a fixed shuffle tree; the result depends only on NB (not on the batch).
__device__ __forceinline__ double warp_sum_partials(const double* __restrict__ p, int NB) {
  const int lane = threadIdx.x & 31;
  double t = 0.0;
  for (int b = lane; b < NB; b += 32) t += p[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// Per sample: total of the NB partials (fixed order). mode 0: store ||g||^2.
// mode 1: relative residual, cycle count and active flag after `inc` cycles, of the active
// samples (of those that `mask` names, if it is given; mask then names those of them that go on).
__global__ void k_norm_update(int B, int NB, const double* __restrict__ partial, double* __restrict__ g2,
                              double* __restrict__ relres, int* __restrict__ cycles, int* __restrict__ active,
                              int mode, int inc, double rtol, int max_cycles, int* __restrict__ n_active,
                              int* __restrict__ mask = nullptr) {
  const int s = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;  // one warp per sample
  if (s >= B) return;
  if (mode == 1 && !(mask ? mask[s] : active[s])) return;
  const double t = warp_sum_partials(partial + (size_t)s * NB, NB);
  if ((threadIdx.x & 31) != 0) return;
  if (mode == 0) {
    g2[s] = t;
    return;
  }
  const double rel = g2[s] > 0.0 ? sqrt(t / g2[s]) : 0.0;
  relres[s] = rel;
  cycles[s] += inc;
  const int c = cycles[s];
  const int still = (rtol > 0.0) ? (rel > rtol && c < max_cycles) : (c < max_cycles);
  active[s] = still;
  if (mask) mask[s] = still;
  if (still) atomicAdd(n_active, 1);
}

// What the red residuals' norm has to exceed for a sample to go on without the full test. Formed
// in the full residual's order of operations (fused = false) they can differ from their part of it
// by the order of the sum alone, so the full test's answer is certain. Formed along with a red pass
// (fused) each is the same eight terms rounded in another order. The two roundings differ by a few
// ulps of the largest term, D u, which grows with (n - 1)^2 and with the contrast of the coefficient:
// about 2^-55 (n - 1)^2 of |g| for one of order one, a sixteenth of the smallest tolerance red_fused
// takes. The eighth on top covers that, not every contrast: on a rough coefficient, within rounding
// of its tolerance, a sample could in principle go on for a cycle that the full test would have
// stopped (never stop early: the full test decides that). It has not been seen: the full residual
// carries the same rounding at the red nodes and the sweep's own at the black ones, so it is the
// larger of the two there (2196 tolerances at and just above the residual of a cycle, variances 1 to
// 9 on grids of 9^3 to 65^3: every solve stopped where the full test stops it). Below those
// tolerances every test is a full one.
__host__ __device__ inline double red_limit(double rtol, bool fused) { return rtol * (fused ? 1.125 : 1.0 + 1e-9); }
inline bool red_fused(double rtol, int n) { return rtol >= 0x1p-51 * (n - 1) * (n - 1); }

// After `inc` more cycles, from the partials of the red residuals alone (a lower bound of the
// norm): a sample whose red residual exceeds `rtol` (red_limit), and which has cycles left, goes on
// (n_active[0]); the others are candidates to stop (cand, n_active[1]), for which the full
// residual decides (k_norm_update).
__global__ void k_norm_red(int B, int NB, const double* __restrict__ partial, const double* __restrict__ g2,
                           int* __restrict__ cycles, const int* __restrict__ active, int* __restrict__ cand, int inc,
                           double rtol, int max_cycles, int* __restrict__ n_active) {
  const int s = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;  // one warp per sample
  if (s >= B) return;
  const bool on = active[s] != 0;
  const double t = on ? warp_sum_partials(partial + (size_t)s * NB, NB) : 0.0;
  if ((threadIdx.x & 31) != 0) return;
  if (!on) {
    cand[s] = 0;
    return;
  }
  const double rel = g2[s] > 0.0 ? sqrt(t / g2[s]) : 0.0;
  const int c = cycles[s] + inc;
  cycles[s] = c;
  const bool go = rel > rtol && c < max_cycles;
  cand[s] = go ? 0 : 1;
  atomicAdd(n_active + (go ? 0 : 1), 1);
}

// g_c = 4 FW(r~) at interior coarse nodes (the coarse boundary of g_c is zeroed once per
// solve and never written).
template <typename T, bool SPLIT_OUT = false>
__global__ void k_restrict(int nf, int B, const T* __restrict__ r, T* __restrict__ gc, const int* __restrict__ active) {
  // nc - 1 = 2^(p-1) = hc: an interior coarse row is X = 1 .. hc - 1
  const int nc = (nf + 1) / 2, hc = nc - 1, lc = 31 - __clz(hc);
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // interior coarse node of a plane
  if (q >= (nc - 2) * hc) return;
  const int X = 1 + (q & (hc - 1)), Y = 1 + (q >> lc);
  if (X > nc - 2) return;
  const size_t nc3 = (size_t)nc * nc * nc, nf3 = (size_t)nf * nf * nf;
  const int nf2 = nf * nf;
  for (int zz = blockIdx.y; zz < B * (nc - 2); zz += gridDim.y) {
    const int s = zz / (nc - 2), Z = 1 + (zz - s * (nc - 2));
    if (active && !active[s]) continue;
    const T* rb = r + (size_t)s * nf3 + (size_t)(2 * Z * nf2 + 2 * Y * nf + 2 * X);
    T v = 0;
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) {
          const T wgt = (T)((2 - abs(dx)) * (2 - abs(dy)) * (2 - abs(dz))) * (T)(1.0 / 16.0);
          v = fma(wgt, rb[dz * nf2 + dy * nf + dx], v);
        }
    if (SPLIT_OUT)
      gc[(size_t)s * split_elems(nc) + split_index(nc, X, Y, Z)] = v;
    else
      gc[(size_t)s * nc3 + (size_t)((Z * nc + Y) * nc + X)] = v;
  }
}

// k_restrict of a residual that is zero at black nodes (k_residual_red): its 13 red terms of
// the 27, in their order.
template <typename T>
__global__ void k_restrict_red(int nf, int B, const T* __restrict__ r, T* __restrict__ gc,
                               const int* __restrict__ active) {
  const int nc = (nf + 1) / 2, hc = nc - 1, lc = 31 - __clz(hc);
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // interior coarse node of a plane
  if (q >= (nc - 2) * hc) return;
  const int X = 1 + (q & (hc - 1)), Y = 1 + (q >> lc);
  if (X > nc - 2) return;
  const size_t nc3 = (size_t)nc * nc * nc, nf3 = (size_t)nf * nf * nf;
  const int nf2 = nf * nf;
  for (int zz = blockIdx.y; zz < B * (nc - 2); zz += gridDim.y) {
    const int s = zz / (nc - 2), Z = 1 + (zz - s * (nc - 2));
    if (active && !active[s]) continue;
    const T* rb = r + (size_t)s * nf3 + (size_t)(2 * Z * nf2 + 2 * Y * nf + 2 * X);
    T v = 0;
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) {
          if ((dx + dy + dz) & 1) continue;
          const T wgt = (T)((2 - abs(dx)) * (2 - abs(dy)) * (2 - abs(dz))) * (T)(1.0 / 16.0);
          v = fma(wgt, rb[dz * nf2 + dy * nf + dx], v);
        }
    gc[(size_t)s * nc3 + (size_t)((Z * nc + Y) * nc + X)] = v;
  }
}

// u_f += trilinear interpolation of e_c at interior fine nodes: a fine node with k odd
// coordinates is the mean of its 2^k coarse neighbours (k = 0: the coincident coarse
// node). Threads of a row take the odd x first and the even x after them, so that a warp
// shares one parity pattern and sums only the distinct neighbours (4.3 instead of 8
// terms per node on average).
template <typename T>
__global__ void k_prolong(int nf, int B, const T* __restrict__ ec, T* __restrict__ u, const int* __restrict__ active) {
  // nf - 1 = 2^p = P: interior x of a row, odd ones (r < P/2: x = 2r + 1) then even ones
  const int nc = (nf + 1) / 2, P = nf - 1, lp = 31 - __clz(P), hp = P >> 1;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= (nf - 2) * P) return;
  const int rr = q & (P - 1), y = 1 + (q >> lp);
  const int x = rr < hp ? 2 * rr + 1 : 2 * (rr - hp) + 2;
  if (x > nf - 2) return;
  const size_t nc3 = (size_t)nc * nc * nc, nf3 = (size_t)nf * nf * nf;
  const int xo = x & 1, yo = y & 1, X = x >> 1, Y = y >> 1;
  for (int zz = blockIdx.y; zz < B * (nf - 2); zz += gridDim.y) {
    const int s = zz / (nf - 2), z = 1 + (zz - s * (nf - 2));
    if (active && !active[s]) continue;
    const int zo = z & 1, Z = z >> 1;
    // the distinct coarse neighbours in the order (Z, Y), (Z, Y+1), (Z+1, Y), (Z+1, Y+1),
    // each row X then X+1, as straight-line code (parities decide which exist)
    const T* r0 = ec + (size_t)s * nc3 + (size_t)((Z * nc + Y) * nc + X);
    T v = 0;
    v += r0[0];
    if (xo) v += r0[1];
    if (yo) {
      v += r0[nc];
      if (xo) v += r0[nc + 1];
    }
    if (zo) {
      const T* r2 = r0 + nc * nc;
      v += r2[0];
      if (xo) v += r2[1];
      if (yo) {
        v += r2[nc];
        if (xo) v += r2[nc + 1];
      }
    }
    const T w = xo + yo + zo == 0 ? T(1) : xo + yo + zo == 1 ? T(0.5) : xo + yo + zo == 2 ? T(0.25) : T(0.125);
    const size_t p = (size_t)s * nf3 + (size_t)((z * nf + y) * nf + x);
    u[p] += w * v;
  }
}

// The sums of k_prolong for the eight fine nodes (2X + dx, 2Y + dy, 2Z + dz) of one coarse
// cell, c = e_c at (X, Y, Z), (X+1, Y, Z), (X, Y+1, Z), (X+1, Y+1, Z), then the same at Z+1:
// every node's sum takes its terms in k_prolong's order, and the nodes whose term
// sequences share a prefix share its partial sum (14 additions for the block instead of 27).
// v[dx + 2 dy + 4 dz].
template <typename T>
__device__ __forceinline__ void prolong_block_sums(const T (&c)[8], T (&v)[8]) {
  T sa = 0;
  sa += c[0];
  const T sab = sa + c[1], sac = sa + c[2];
  const T sabcd = (sab + c[2]) + c[3];
  v[0] = sa;
  v[1] = sab;
  v[2] = sac;
  v[3] = sabcd;
  v[4] = sa + c[4];
  v[5] = (sab + c[4]) + c[5];
  v[6] = (sac + c[4]) + c[6];
  v[7] = (((sabcd + c[4]) + c[5]) + c[6]) + c[7];
}

// k_prolong's result (bit for bit) with one thread per coarse cell: the eight fine nodes
// (2X + dx, 2Y + dy, 2Z + dz) of the cell, their sums from prolong_block_sums, u += w v at
// the interior ones. Every thread runs the same operations (no parity divergence) and the
// block shares partial sums: 2.75 instead of 4.4 FP64 operations per fine node. Grid: coarse
// cells of a plane, (sample, cell plane) planes. BLACK: the black nodes (dx + dy + dz odd)
// only, 1.6 operations per fine node: a red pass follows, which overwrites the red nodes
// without reading them (the compiler drops the sums no black node needs).
template <typename T, bool BLACK = false>
__global__ void __launch_bounds__(128) k_prolong_blk(int nf, int B, const T* __restrict__ ec, T* __restrict__ u,
                                                     const int* __restrict__ active) {
  const int nc = (nf + 1) / 2, mc = nc - 1;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= mc * mc) return;
  const int Y = q / mc, X = q - Y * mc;
  const size_t nc3 = (size_t)nc * nc * nc, nf3 = (size_t)nf * nf * nf, nc2 = (size_t)nc * nc;
  for (int zz = blockIdx.y; zz < B * mc; zz += gridDim.y) {
    const int s = zz / mc, Z = zz - s * mc;
    if (active && !active[s]) continue;
    const T* e = ec + (size_t)s * nc3 + (size_t)((Z * nc + Y) * nc + X);
    const T c[8] = {e[0], e[1], e[nc], e[nc + 1], e[nc2], e[nc2 + 1], e[nc2 + nc], e[nc2 + nc + 1]};
    T v[8];
    prolong_block_sums(c, v);
    T* ub = u + (size_t)s * nf3;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int dx = k & 1, dy = (k >> 1) & 1, dz = k >> 2;
      if (BLACK && !((dx + dy + dz) & 1)) continue;
      const int x = 2 * X + dx, y = 2 * Y + dy, z = 2 * Z + dz;
      if (x < 1 || y < 1 || z < 1 || x > nf - 2 || y > nf - 2 || z > nf - 2) continue;
      const T w = dx + dy + dz == 0 ? T(1) : dx + dy + dz == 1 ? T(0.5) : dx + dy + dz == 2 ? T(0.25) : T(0.125);
      ub[(size_t)((z * nf + y) * nf + x)] += w * v[k];
    }
  }
}

// k_prolong_blk on colour-split storage of both grids (LG: the fine grid's). Fine node
// (2X + dx, ...) is colour (dx + dy + dz) & 1, slot X; coarse (X', Y', Z') colour
// (X' + Y' + Z') & 1, slot X' / 2. Grid (coarse cells of a plane, cell planes, samples).
// BLACK: as in k_prolong_blk.
template <int LG, typename T, bool BLACK = false>
__global__ void __launch_bounds__(128) k_prolong_blk_split(const T* __restrict__ ec, T* __restrict__ u,
                                                           const int* __restrict__ active) {
  using F = SplitGeo<LG>;
  using C = SplitGeo<LG - 1>;
  constexpr int mc = C::n - 1;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= mc * mc) return;
  const int s = blockIdx.z;
  if (active && !active[s]) return;
  const int Y = q / mc, X = q - Y * mc, Z = (int)blockIdx.y;
  const T* e = ec + (size_t)s * C::NS;
  auto at = [&](int i, int j, int k) -> T {
    const int xx = X + i, yy = Y + j, zz = Z + k;
    return e[(size_t)((xx + yy + zz) & 1) * C::BLK + (size_t)((zz * C::n + yy) * C::P + (xx >> 1))];
  };
  const T c[8] = {at(0, 0, 0), at(1, 0, 0), at(0, 1, 0), at(1, 1, 0), at(0, 0, 1), at(1, 0, 1), at(0, 1, 1), at(1, 1, 1)};
  T v[8];
  prolong_block_sums(c, v);
  T* ub = u + (size_t)s * F::NS;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int dx = k & 1, dy = (k >> 1) & 1, dz = k >> 2;
    if (BLACK && !((dx + dy + dz) & 1)) continue;
    const int x = 2 * X + dx, y = 2 * Y + dy, z = 2 * Z + dz;
    if (x < 1 || y < 1 || z < 1 || x > F::n - 2 || y > F::n - 2 || z > F::n - 2) continue;
    const T w = dx + dy + dz == 0 ? T(1) : dx + dy + dz == 1 ? T(0.5) : dx + dy + dz == 2 ? T(0.25) : T(0.125);
    ub[(size_t)((dx + dy + dz) & 1) * F::BLK + (size_t)((z * F::n + y) * F::P + X)] += w * v[k];
  }
}

// g = h^2 f (f == NULL: h^2) on interior nodes, 0 on the boundary; u boundary := 0.
template <bool SPLIT = false>
__global__ void k_prepare(int n, int B, double h2, const double* __restrict__ f, double* __restrict__ g,
                          double* __restrict__ u) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // node of the plane
  if (q >= n * n) return;
  const int y = q / n, x = q - y * n;
  const size_t n3 = (size_t)n * n * n;
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, z = zz - s * n;
    const size_t tp = (size_t)s * n3 + (size_t)(z * n * n + q), t = SPLIT ? node_at<true>(n, s, x, y, z) : tp;
    const bool in = x > 0 && y > 0 && z > 0 && x < n - 1 && y < n - 1 && z < n - 1;
    g[t] = in ? h2 * (f ? f[tp] : 1.0) : 0.0;
    if (!in) u[t] = 0.0;
  }
}

// Mixed refinement update u64 += e32 at interior nodes of active samples (SPLIT: e in
// colour-split storage).
template <bool SPLIT>
__global__ void k_update_mixed(int n, int B, const float* __restrict__ e, double* __restrict__ u,
                               const int* __restrict__ active) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // node of the plane
  if (q >= n * n) return;
  const int y = q / n, x = q - y * n;
  const size_t n3 = (size_t)n * n * n;
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, z = zz - s * n;
    if (!active[s]) continue;
    const size_t t = (size_t)s * n3 + (size_t)(z * n * n + q);
    const float ev = SPLIT ? e[(size_t)s * split_elems(n) + split_index(n, x, y, z)] : e[t];
    u[t] += widen(ev);  // e is zero on the boundary
  }
}

// QoI partial sums (trapezoid weights, Kahan in each thread). Grid (NB, B).
__global__ void __launch_bounds__(kThreads) k_qoi(int n, const double* __restrict__ u, double* __restrict__ partial) {
  const int s = blockIdx.y;
  const int lo = (n - 1) / 4, S = (n - 1) / 2 + 1;
  const unsigned S3 = (unsigned)S * S * S, S2 = (unsigned)S * S, uS = (unsigned)S;
  const size_t n3 = (size_t)n * n * n;
  const unsigned chunk = (S3 + gridDim.x - 1) / gridDim.x;
  const unsigned a = blockIdx.x * chunk, b = a + chunk < S3 ? a + chunk : S3;
  double sum = 0.0, comp = 0.0;
  for (unsigned i = a + threadIdx.x; i < b; i += kThreads) {
    const unsigned czq = i / S2, rem = i - czq * S2, cyq = rem / uS;
    const int cz = (int)czq, cy = (int)cyq, cx = (int)(rem - cyq * uS);
    const double w = (cx == 0 || cx == S - 1 ? 0.5 : 1.0) * (cy == 0 || cy == S - 1 ? 0.5 : 1.0) *
                     (cz == 0 || cz == S - 1 ? 0.5 : 1.0);
    const double v = w * u[(size_t)s * n3 + ((size_t)(lo + cz) * n + (lo + cy)) * n + (lo + cx)];
    const double yk = v - comp;
    const double tk = sum + yk;
    comp = (tk - sum) - yk;
    sum = tk;
  }
  const double tot = block_sum<kThreads>(sum);
  if (threadIdx.x == 0) partial[(size_t)s * gridDim.x + blockIdx.x] = tot;
}

__global__ void k_qoi_final(int B, int NB, double scale, const double* __restrict__ partial, double* __restrict__ Q) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= B) return;
  double t = 0.0;
  for (int b = 0; b < NB; ++b) t += partial[(size_t)s * NB + b];
  Q[s] = scale * t;
}

// ---------------------------------------------------------------------------------
// P1 finite elements on the tetrahedral mesh (Sec. 3.1): every grid cube is cut into the
// six tetrahedra {O, O + e_a, O + e_a + e_b, O + (1,1,1)}; the stiffness with the four-vertex
// quadrature of k couples only the axis edges of each element's vertex path (the
// barycentric gradients of the path's non-adjacent vertices are orthogonal), so the
// operator keeps the seven-point form with, per axis edge, the mean over the six elements
// that share it of their vertex-mean coefficient kbar:
//   K_a(P) = (k_P + k_{P+a}) / 4 + (k_{P+a+b} + k_{P+a+c} + k_{P+a+b+c} + k_{P-b} + k_{P-c}
//            + k_{P-b-c}) / 12      ({a, b, c} = {x, y, z}),
// in the h^2-scaled form (FE matrix / h); the load of f = 1 is h^3 per interior node, the
// g = h^2 f of the scaled form. split: the faces go straight to colour-split storage (assembled in
// plain arrays and copied, a 65^3 / 33^3 FMG level of 108 samples took 0.9 of its 17.6 ms longer).
// ---------------------------------------------------------------------------------
template <typename T>
__global__ void k_faces_fe(const double* __restrict__ k0, int n0, int st0, int n, int B, T* __restrict__ Kx,
                           T* __restrict__ Ky, T* __restrict__ Kz, int split = 0) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // node of the plane
  if (q >= n * n) return;
  const int y = q / n, x = q - y * n;
  const size_t n3 = (size_t)n * n * n, n03 = (size_t)n0 * n0 * n0;
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, z = zz - s * n;
    const double* kb = k0 + (size_t)s * n03;
    auto K = [&](int dx, int dy, int dz) {
      return kb[((size_t)(st0 * (z + dz)) * n0 + (size_t)(st0 * (y + dy))) * n0 + (size_t)(st0 * (x + dx))];
    };
    const bool ix = x >= 1 && x <= n - 2, iy = y >= 1 && y <= n - 2, iz = z >= 1 && z <= n - 2;
    const size_t t = split ? (size_t)s * split_elems(n) + split_index(n, x, y, z) : (size_t)s * n3 + (size_t)(z * n * n + q);
    double fx = 0.0, fy = 0.0, fz = 0.0;
    if (x <= n - 2 && iy && iz)
      fx = (K(0, 0, 0) + K(1, 0, 0)) * 0.25 +
           (K(1, 1, 0) + K(1, 0, 1) + K(1, 1, 1) + K(0, -1, 0) + K(0, 0, -1) + K(0, -1, -1)) * (1.0 / 12.0);
    if (y <= n - 2 && ix && iz)
      fy = (K(0, 0, 0) + K(0, 1, 0)) * 0.25 +
           (K(0, 1, 1) + K(1, 1, 0) + K(1, 1, 1) + K(0, 0, -1) + K(-1, 0, 0) + K(-1, 0, -1)) * (1.0 / 12.0);
    if (z <= n - 2 && ix && iy)
      fz = (K(0, 0, 0) + K(0, 0, 1)) * 0.25 +
           (K(1, 0, 1) + K(0, 1, 1) + K(1, 1, 1) + K(-1, 0, 0) + K(0, -1, 0) + K(-1, -1, 0)) * (1.0 / 12.0);
    Kx[t] = (T)fx;
    Ky[t] = (T)fy;
    Kz[t] = (T)fz;
  }
}

// P1 interpolation between nested tetrahedral meshes, added on interior fine nodes: a
// fine node with odd coordinates d (a 0/1 vector) is the midpoint of the coarse edge from
// c0 = (f - d) / 2 to c0 + d (a mesh edge: every direction e_a, e_a + e_b, (1,1,1) is
// one), so it takes the mean of the two; a node with d = 0 is a coarse node.
template <typename T, bool SPLIT = false>
__global__ void k_prolong_p1(int nf, int B, const T* __restrict__ ec, T* __restrict__ u,
                             const int* __restrict__ active) {
  const int m = nf - 2, nc = (nf + 1) / 2;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // interior node of the plane
  if (q >= m * m) return;
  const int y = 1 + q / m, x = 1 + q - (y - 1) * m;
  for (int zz = blockIdx.y; zz < B * m; zz += gridDim.y) {
    const int s = zz / m, z = 1 + zz - s * m;
    if (active && !active[s]) continue;
    const int dx = x & 1, dy = y & 1, dz = z & 1;
    const int X0 = (x - dx) >> 1, Y0 = (y - dy) >> 1, Z0 = (z - dz) >> 1;
    T v = ec[node_at<SPLIT>(nc, s, X0, Y0, Z0)];
    if (dx | dy | dz) v = T(0.5) * (v + ec[node_at<SPLIT>(nc, s, X0 + dx, Y0 + dy, Z0 + dz)]);
    u[node_at<SPLIT>(nf, s, x, y, z)] += v;
  }
}

// Its transpose on interior coarse nodes, scaled for the coarse h^2-scaled system:
// g_c = (h / h_c) P^T r = (1/2) (r(2c) + (1/2) sum over the 14 mesh-edge directions d of
// r(2c + d)) (the fine residual r is zero on the boundary).
template <typename T, bool SPLIT = false>
__global__ void k_restrict_p1(int nf, int B, const T* __restrict__ r, T* __restrict__ gc,
                              const int* __restrict__ active) {
  const int nc = (nf + 1) / 2, mc = nc - 2;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // interior coarse node of the plane
  if (q >= mc * mc) return;
  const int Y = 1 + q / mc, X = 1 + q - (Y - 1) * mc;
  for (int zz = blockIdx.y; zz < B * mc; zz += gridDim.y) {
    const int s = zz / mc, Z = 1 + zz - s * mc;
    if (active && !active[s]) continue;
    auto R = [&](int dx, int dy, int dz) { return r[node_at<SPLIT>(nf, s, 2 * X + dx, 2 * Y + dy, 2 * Z + dz)]; };
    T acc = R(-1, 0, 0) + R(1, 0, 0);
    acc += R(0, -1, 0) + R(0, 1, 0);
    acc += R(0, 0, -1) + R(0, 0, 1);
    acc += R(-1, -1, 0) + R(1, 1, 0);
    acc += R(0, -1, -1) + R(0, 1, 1);
    acc += R(-1, 0, -1) + R(1, 0, 1);
    acc += R(-1, -1, -1) + R(1, 1, 1);
    gc[node_at<SPLIT>(nc, s, X, Y, Z)] = T(0.5) * R(0, 0, 0) + T(0.25) * acc;
  }
}

// k_prolong_p1 at the black fine nodes only (a red pass follows, which overwrites the red
// nodes without reading them); a black node has an odd number of odd coordinates, so it is
// always the midpoint of a coarse edge. Threads enumerate rows of black nodes.
template <typename T, bool SPLIT>
__global__ void k_prolong_p1_black(int nf, int B, const T* __restrict__ ec, T* __restrict__ u,
                                   const int* __restrict__ active) {
  const int m = nf - 2, nc = (nf + 1) / 2, half = nc - 1;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= m * half) return;
  const int y = 1 + q / half, xi = q - (y - 1) * half;
  for (int zz = blockIdx.y; zz < B * m; zz += gridDim.y) {
    const int s = zz / m, z = 1 + zz - s * m;
    if (active && !active[s]) continue;
    const int x = 1 + 2 * xi + ((y + z) & 1);
    if (x > nf - 2) continue;
    const int dx = x & 1, dy = y & 1, dz = z & 1;
    const int X0 = (x - dx) >> 1, Y0 = (y - dy) >> 1, Z0 = (z - dz) >> 1;
    u[node_at<SPLIT>(nf, s, x, y, z)] +=
        T(0.5) * (ec[node_at<SPLIT>(nc, s, X0, Y0, Z0)] + ec[node_at<SPLIT>(nc, s, X0 + dx, Y0 + dy, Z0 + dz)]);
  }
}

// k_restrict_p1 of a residual that is zero at black nodes (k_residual_red): the six diagonal
// directions of the faces and the node itself.
template <typename T, bool SPLIT>
__global__ void k_restrict_p1_red(int nf, int B, const T* __restrict__ r, T* __restrict__ gc,
                                  const int* __restrict__ active) {
  const int nc = (nf + 1) / 2, mc = nc - 2;
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // interior coarse node of the plane
  if (q >= mc * mc) return;
  const int Y = 1 + q / mc, X = 1 + q - (Y - 1) * mc;
  for (int zz = blockIdx.y; zz < B * mc; zz += gridDim.y) {
    const int s = zz / mc, Z = 1 + zz - s * mc;
    if (active && !active[s]) continue;
    auto R = [&](int dx, int dy, int dz) { return r[node_at<SPLIT>(nf, s, 2 * X + dx, 2 * Y + dy, 2 * Z + dz)]; };
    T acc = R(-1, -1, 0) + R(1, 1, 0);
    acc += R(0, -1, -1) + R(0, 1, 1);
    acc += R(-1, 0, -1) + R(1, 0, 1);
    gc[node_at<SPLIT>(nc, s, X, Y, Z)] = T(0.5) * R(0, 0, 0) + T(0.25) * acc;
  }
}

// Q[s] = u(1/4, 1/4, 1/4) (a node: (n - 1) / 4 in every coordinate).
__global__ void k_qoi_point(int n, int B, const double* __restrict__ u, double* __restrict__ Q) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= B) return;
  const int c = (n - 1) / 4;
  Q[s] = u[(size_t)s * n * n * n + ((size_t)c * n + c) * n + c];
}

// Flux of k du/dx_2 across x_2 = 1/4 as the mean over the layer of elements between
// x_2 = 1/4 - h and 1/4: per cube of the layer (origin y = (n-1)/4 - 1) and each of its
// six elements (path a, b, c), kbar times the difference of u along the path's y step;
// per-block partial sums (grid (NB, B)), scaled by h/6 in k_qoi_final. k from the FP64
// field k0 (stride st0).
__global__ void __launch_bounds__(kThreads) k_qoi_flux(int n, const double* __restrict__ u,
                                                       const double* __restrict__ k0, int n0, int st0,
                                                       double* __restrict__ partial) {
  const int s = blockIdx.y, NB = gridDim.x;
  const int m = n - 1, j0 = (n - 1) / 4 - 1;
  const size_t n3 = (size_t)n * n * n, n03 = (size_t)n0 * n0 * n0;
  const double* ub = u + (size_t)s * n3;
  const double* kb = k0 + (size_t)s * n03;
  double acc = 0.0;
  for (int c = blockIdx.x * kThreads + threadIdx.x; c < m * m; c += NB * kThreads) {
    const int zc = c / m, xc = c - zc * m;
    double uv[8], kv[8];  // cube corners, bit 0 = x, bit 1 = y, bit 2 = z
    for (int v = 0; v < 8; ++v) {
      const int X = xc + (v & 1), Y = j0 + ((v >> 1) & 1), Z = zc + (v >> 2);
      uv[v] = ub[((size_t)Z * n + Y) * n + X];
      kv[v] = kb[((size_t)(st0 * Z) * n0 + (size_t)(st0 * Y)) * n0 + (size_t)(st0 * X)];
    }
    const int ax[6][3] = {{0, 1, 2}, {0, 2, 1}, {1, 0, 2}, {1, 2, 0}, {2, 0, 1}, {2, 1, 0}};
    for (int e = 0; e < 6; ++e) {
      int v = 0, vs[4];
      vs[0] = 0;
      double dy = 0.0;
      for (int i = 0; i < 3; ++i) {
        const int w = v | (1 << ax[e][i]);
        if (ax[e][i] == 1) dy = uv[w] - uv[v];
        v = w;
        vs[i + 1] = v;
      }
      const double kbar = 0.25 * (kv[vs[0]] + kv[vs[1]] + kv[vs[2]] + kv[vs[3]]);
      acc = fma(kbar, dy, acc);
    }
  }
  const double b = block_sum<kThreads>(acc);
  if (threadIdx.x == 0) partial[(size_t)s * NB + blockIdx.x] = b;
}

// ---------------------------------------------------------------------------------
// Flexible preconditioned conjugate gradients (FP64 recurrences; the V-cycle is the
// preconditioner). All vectors are FP64 on the finest grid; per-sample scalars.
// ---------------------------------------------------------------------------------

// True in every thread of the block of a sample's grid that finishes last: `total` blocks count
// themselves in *tick, which the last one resets for the next kernel. Thread 0 has written the
// block's partials before the call. The last block then does the per-sample scalar work, so no
// launch of its own is needed for it.
__device__ __forceinline__ bool last_block(int* tick, int total) {
  __shared__ int last;
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(tick, 1) == total - 1;
    if (last) *tick = 0;
    __threadfence();
  }
  __syncthreads();
  return last != 0;
}
// warp_sum_partials of partials that other blocks of this launch wrote (read past the L1)
__device__ __forceinline__ double warp_sum_fresh(const double* p, int NB) {
  double t = 0.0;
#pragma unroll 4
  for (int b = threadIdx.x & 31; b < NB; b += 32) t += __ldcg(p + b);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// q = A~ p on interior nodes (0 on the boundary): v = D p, then the six faces in the order
// -x, +x, -y, +y, -z, +z, and partials of p.q, by column z-marches: a thread owns one
// (x, y) column of a z-slab and carries p and Kz of the planes below and above in
// registers (11 loads per node), FP32 faces widened on the integer pipe. Grid (column blocks, z-slabs, B), 128 threads; one partial of p.q per
// (column block, slab), a partition fixed by n (apply_slabs).
template <typename TK, typename TD>
__global__ void __launch_bounds__(128)
    k_apply_dot_z(int n, int zslab, const TK* __restrict__ Kx, const TK* __restrict__ Ky, const TK* __restrict__ Kz,
                  const TD* __restrict__ D, const double* __restrict__ p, double* __restrict__ q,
                  double* __restrict__ partial, const int* __restrict__ active) {
  const int s = blockIdx.z;
  if (!active[s]) return;
  const int nb = gridDim.x * gridDim.y, b = blockIdx.y * gridDim.x + blockIdx.x;
  const int c = blockIdx.x * 128 + threadIdx.x;  // column y n + x
  const int zlo = 1 + blockIdx.y * zslab, zhi = min(n - 2, zlo + zslab - 1);
  const size_t n2 = (size_t)n * n;
  double acc = 0.0;
  if (c < n * n) {
    const int y = c / n, x = c - y * n;
    const size_t col = (size_t)s * n2 * n + c;
    if (x > 0 && y > 0 && x < n - 1 && y < n - 1) {
      double pm = p[col + (size_t)(zlo - 1) * n2], pc = p[col + (size_t)zlo * n2];
      double kzm = widen(Kz[col + (size_t)(zlo - 1) * n2]);
      for (int z = zlo; z <= zhi; ++z) {
        const size_t t = col + (size_t)z * n2;
        const double pp = p[t + n2];
        const double kzp = widen(Kz[t]);
        double v = widen(D[t]) * pc;
        v = fma(-widen(Kx[t - 1]), p[t - 1], v);
        v = fma(-widen(Kx[t]), p[t + 1], v);
        v = fma(-widen(Ky[t - n]), p[t - n], v);
        v = fma(-widen(Ky[t]), p[t + n], v);
        v = fma(-kzm, pm, v);
        v = fma(-kzp, pp, v);
        acc = fma(pc, v, acc);
        q[t] = v;
        pm = pc;
        pc = pp;
        kzm = kzp;
      }
    } else {
      for (int z = zlo; z <= zhi; ++z) q[col + (size_t)z * n2] = 0.0;
    }
    if (blockIdx.y == 0) q[col] = 0.0;                                    // plane z = 0
    if (blockIdx.y == gridDim.y - 1) q[col + (size_t)(n - 1) * n2] = 0.0;  // plane z = n-1
  }
  const double bs = block_sum<128>(acc);
  if (threadIdx.x == 0) partial[(size_t)s * nb + b] = bs;
}

// alpha = rz / p.q from k_apply_dot_z's partials, one warp per sample.
__global__ void k_cg_alpha(int B, int NB, const double* __restrict__ part, const double* __restrict__ rz,
                           double* __restrict__ alpha, const int* __restrict__ active) {
  const int s = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (s >= B || !active[s]) return;
  const double t = warp_sum_partials(part + (size_t)s * NB, NB);
  if ((threadIdx.x & 31) == 0) alpha[s] = t != 0.0 ? rz[s] / t : 0.0;
}

// z-slabs of the column z-march kernels: a function of n only (so a sample's sums do not
// depend on the batch): enough (column, slab) threads to fill the GPU for one sample, but
// slabs of at least 8 planes, so that carrying the planes below and above in registers
// saves loads (one-plane slabs would load more than the flat kernels).
inline int apply_slabs(int n, int* zslab) {
  int slabs = (int)((131072LL + (long long)n * n - 1) / ((long long)n * n));
  const int deep = (n - 2) / 8 > 1 ? (n - 2) / 8 : 1;
  if (slabs > deep) slabs = deep;
  if (slabs < 1) slabs = 1;
  *zslab = (n - 2 + slabs - 1) / slabs;
  return (n - 2 + *zslab - 1) / *zslab;
}
inline int apply_blocks(int n) {
  int zs = 0;
  return ((n * n + 127) / 128) * apply_slabs(n, &zs);
}

// r~ = g - D u + sum K u_q on interior nodes (0 on the boundary) by column z-marches (the
// launch shape and partition of k_apply_dot_z): rr = g - D u, then the faces in the order
// -x, +x, -y, +y, -z, +z; optional store of r~ (type TR) and per-(column block, slab)
// partials of r~^2 (FP64).
template <typename T, typename TD, typename TU, typename TR, bool SPLIT_OUT = false>
__global__ void __launch_bounds__(128)
    k_residual_z(int n, int zslab, const T* __restrict__ Kx, const T* __restrict__ Ky, const T* __restrict__ Kz,
                 const TD* __restrict__ D, const TD* __restrict__ g, const TU* __restrict__ u, TR* __restrict__ r,
                 double* __restrict__ partial, const int* __restrict__ active) {
  const int s = blockIdx.z;
  if (active && !active[s]) return;
  const int nb = gridDim.x * gridDim.y, b = blockIdx.y * gridDim.x + blockIdx.x;
  const int c = blockIdx.x * 128 + threadIdx.x;  // column y n + x
  const int zlo = 1 + blockIdx.y * zslab, zhi = min(n - 2, zlo + zslab - 1);
  const size_t n2 = (size_t)n * n;
  double sq = 0.0;
  // store index of r~ at plane z of this column
  const int cy = c < n * n ? c / n : 0, cx = c - cy * n;
  auto rix = [&](size_t t, int z) -> size_t {
    return SPLIT_OUT ? (size_t)s * split_elems(n) + split_index(n, cx, cy, z) : t;
  };
  if (c < n * n) {
    const int y = cy, x = cx;
    const size_t col = (size_t)s * n2 * n + c;
    if (x > 0 && y > 0 && x < n - 1 && y < n - 1) {
      TD um = to_t<TD>(u[col + (size_t)(zlo - 1) * n2]), uc = to_t<TD>(u[col + (size_t)zlo * n2]);
      TD kzm = to_t<TD>(Kz[col + (size_t)(zlo - 1) * n2]);
      for (int z = zlo; z <= zhi; ++z) {
        const size_t t = col + (size_t)z * n2;
        const TD up = to_t<TD>(u[t + n2]);
        const TD kzp = to_t<TD>(Kz[t]);
        TD rr = fma(-D[t], uc, g[t]);
        rr = fma(to_t<TD>(Kx[t - 1]), to_t<TD>(u[t - 1]), rr);
        rr = fma(to_t<TD>(Kx[t]), to_t<TD>(u[t + 1]), rr);
        rr = fma(to_t<TD>(Ky[t - n]), to_t<TD>(u[t - n]), rr);
        rr = fma(to_t<TD>(Ky[t]), to_t<TD>(u[t + n]), rr);
        rr = fma(kzm, um, rr);
        rr = fma(kzp, up, rr);
        if (r) r[rix(t, z)] = (TR)rr;
        sq += (double)rr * (double)rr;
        um = uc;
        uc = up;
        kzm = kzp;
      }
    } else if (r) {
      for (int z = zlo; z <= zhi; ++z) r[rix(col + (size_t)z * n2, z)] = TR(0);
    }
    if (r && blockIdx.y == 0) r[rix(col, 0)] = TR(0);                                          // plane z = 0
    if (r && blockIdx.y == gridDim.y - 1) r[rix(col + (size_t)(n - 1) * n2, n - 1)] = TR(0);  // plane z = n-1
  }
  if (partial) {
    const double bs = block_sum<128>(sq);
    if (threadIdx.x == 0) partial[(size_t)s * nb + b] = bs;
  }
}

// The convergence residual of an FP64 colour-split grid: k_residual_z's column z-march,
// launch shape and partition (partials of r~^2 per (column block, slab)), reading the
// split storage; nothing stored. Grid (column blocks, z-slabs, samples), 128 threads.
__global__ void __launch_bounds__(128)
    k_residual_norm_split(int n, int zslab, const double* __restrict__ Kx, const double* __restrict__ Ky,
                          const double* __restrict__ Kz, const double* __restrict__ D, const double* __restrict__ g,
                          const double* __restrict__ u, double* __restrict__ partial, const int* __restrict__ active) {
  const int s = blockIdx.z;
  if (active && !active[s]) return;
  const int nb = gridDim.x * gridDim.y, b = blockIdx.y * gridDim.x + blockIdx.x;
  const int c = blockIdx.x * 128 + threadIdx.x;
  const int zlo = 1 + blockIdx.y * zslab, zhi = min(n - 2, zlo + zslab - 1);
  const size_t base = (size_t)s * split_elems(n);
  double sq = 0.0;
  if (c < n * n) {
    const int y = c / n, x = c - y * n;
    if (x > 0 && y > 0 && x < n - 1 && y < n - 1) {
      auto at = [&](int xx, int yy, int zz) -> size_t { return base + split_index(n, xx, yy, zz); };
      double um = u[at(x, y, zlo - 1)], uc = u[at(x, y, zlo)];
      double kzm = Kz[at(x, y, zlo - 1)];
      for (int z = zlo; z <= zhi; ++z) {
        const size_t t = at(x, y, z);
        const double up = u[at(x, y, z + 1)];
        const double kzp = Kz[t];
        double rr = fma(-D[t], uc, g[t]);
        rr = fma(Kx[at(x - 1, y, z)], u[at(x - 1, y, z)], rr);
        rr = fma(Kx[t], u[at(x + 1, y, z)], rr);
        rr = fma(Ky[at(x, y - 1, z)], u[at(x, y - 1, z)], rr);
        rr = fma(Ky[t], u[at(x, y + 1, z)], rr);
        rr = fma(kzm, um, rr);
        rr = fma(kzp, up, rr);
        sq += (double)rr * (double)rr;
        um = uc;
        uc = up;
        kzm = kzp;
      }
    }
  }
  const double bs = block_sum<128>(sq);
  if (threadIdx.x == 0) partial[(size_t)s * nb + b] = bs;
}

// Partials of r~^2 over the red nodes only (k_residual_red's operations), for the convergence
// test after a cycle that ends on a black pass: the black residuals are zero up to rounding, so
// half the work decides whether a sample goes on. Bound by the FP64 pipe (8 operations per red
// node). A thread takes one red slot of a plane (the split form a pair of slots on 16-byte
// loads) through a z-slab; the partition is a function of n only. Grid (slot blocks, z-slabs,
// samples), 128 threads. (Plain storage; the split form below takes the test along with the next
// cycle's first red pass.)
template <typename T>
__global__ void __launch_bounds__(128)
    k_norm_red_z(int n, int zslab, const T* __restrict__ Kx, const T* __restrict__ Ky, const T* __restrict__ Kz,
                 const T* __restrict__ D, const T* __restrict__ g, const T* __restrict__ u,
                 double* __restrict__ partial, const int* __restrict__ active) {
  const int s = blockIdx.z;
  if (!active[s]) return;
  const int m = n - 2, half = (n - 1) / 2;
  const int q = blockIdx.x * 128 + threadIdx.x;
  const int zlo = 1 + blockIdx.y * zslab, zhi = min(n - 2, zlo + zslab - 1);
  const size_t n2 = (size_t)n * n;
  double sq = 0.0;
  if (q < m * half) {
    const int yi = q / half, xi = q - yi * half, y = 1 + yi;
    for (int z = zlo; z <= zhi; ++z) {
      const int x = 1 + ((y + z + 1) & 1) + 2 * xi;
      if (x > n - 2) continue;
      const size_t p = (size_t)s * n2 * n + (size_t)(z * n * n + y * n + x);
      T rr = fma(-D[p], u[p], g[p]);
      rr = fma(Kx[p - 1], u[p - 1], rr);
      rr = fma(Kx[p], u[p + 1], rr);
      rr = fma(Ky[p - n], u[p - n], rr);
      rr = fma(Ky[p], u[p + n], rr);
      rr = fma(Kz[p - n2], u[p - n2], rr);
      rr = fma(Kz[p], u[p + n2], rr);
      sq += (double)rr * (double)rr;
    }
  }
  const double b = block_sum<128>(sq);
  if (threadIdx.x == 0) partial[((size_t)s * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = b;
}

// The next cycle's first red pass (k_rbgs_split64's operations) on colour-split storage with the
// red residuals it passes by: with acc = g + sum K u_q, the residual is acc - D u and the update
// acc / D, so the test costs two FP64 operations per red node instead of eight (212 us a launch on a
// 129^3 / 65^3 level of 24 samples, 0.93 TFLOP/s; the pass alone 150, the test alone 184). The replaced red
// values go to `old` (one colour block per sample) for the samples that turn out to be done
// (k_restore_red).
template <int LG>
__global__ void __launch_bounds__(128)
    k_rbgs_norm_split(int zslab, const double* __restrict__ Kx, const double* __restrict__ Ky,
                      const double* __restrict__ Kz, const double* __restrict__ D, const double* __restrict__ Dinv,
                      const double* __restrict__ g, double* __restrict__ u, double* __restrict__ old,
                      double* __restrict__ partial, const int* __restrict__ active) {
  using G = SplitGeo<LG>;
  const int s = blockIdx.z;
  if (!active[s]) return;
  const int q = blockIdx.x * 128 + threadIdx.x;
  const int zlo = 1 + blockIdx.y * zslab, zhi = min(G::n - 2, zlo + zslab - 1);
  const size_t cb = (size_t)s * G::NS, ob = cb + G::BLK;
  double sq = 0.0;
  if (q < G::m * G::A2) {
    const int yi = q / G::A2, qi = q - yi * G::A2, y = 1 + yi, xi0 = 2 * qi;
    for (int z = zlo; z <= zhi; ++z) {
      const int par = (y + z) & 1, x0 = 2 * xi0 + par;
      if (x0 > G::n - 2) continue;
      const int o = (z * G::n + y) * G::P + xi0;
      const double2 kx2 = ld2(Kx + cb + o), ky2 = ld2(Ky + cb + o), kz2 = ld2(Kz + cb + o);
      const double2 d2 = ld2(D + cb + o), di2 = ld2(Dinv + cb + o), g2 = ld2(g + cb + o), up2 = ld2(u + cb + o);
      const double* uo = u + ob;
      const double2 kxm2 = ld2(Kx + ob + o), kym2 = ld2(Ky + ob + o - G::P), kzm2 = ld2(Kz + ob + o - G::NP);
      const double2 um2 = ld2(uo + o), uym2 = ld2(uo + o - G::P), uyp2 = ld2(uo + o + G::P);
      const double2 uzm2 = ld2(uo + o - G::NP), uzp2 = ld2(uo + o + G::NP);
      double kext = 0.0, uext = 0.0;
      if (par) {
        uext = uo[o + 2];
      } else if (x0 > 0) {
        kext = Kx[ob + o - 1];
        uext = uo[o - 1];
      }
      *reinterpret_cast<double2*>(old + (size_t)s * G::BLK + o) = up2;
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (x0 + 2 * i < 1 || x0 + 2 * i > G::n - 2) continue;
        const double kl = par ? comp2(kxm2, i) : (i == 0 ? kext : comp2(kxm2, i - 1));
        const double ul = par ? comp2(um2, i) : (i == 0 ? uext : comp2(um2, i - 1));
        const double ur = par ? (i == 1 ? uext : comp2(um2, i + 1)) : comp2(um2, i);
        double acc = comp2(g2, i);
        acc = fma(kl, ul, acc);
        acc = fma(comp2(kx2, i), ur, acc);
        acc = fma(comp2(kym2, i), comp2(uym2, i), acc);
        acc = fma(comp2(ky2, i), comp2(uyp2, i), acc);
        acc = fma(comp2(kzm2, i), comp2(uzm2, i), acc);
        acc = fma(comp2(kz2, i), comp2(uzp2, i), acc);
        const double rr = fma(-comp2(d2, i), comp2(up2, i), acc);
        sq = fma(rr, rr, sq);
        u[cb + o + i] = acc * comp2(di2, i);
      }
    }
  }
  const double b = block_sum<128>(sq);
  if (threadIdx.x == 0) partial[((size_t)s * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = b;
}

// Puts back the interior red values that k_rbgs_norm_split replaced, for the samples in `cand`.
// Grid (two-slot groups of the interior rows of a plane, interior planes, samples).
template <int LG>
__global__ void __launch_bounds__(128) k_restore_red(const double* __restrict__ old, double* __restrict__ u,
                                                     const int* __restrict__ cand) {
  using G = SplitGeo<LG>;
  const int s = blockIdx.z, q = blockIdx.x * 128 + threadIdx.x;
  if (!cand[s] || q >= G::m * G::A2) return;
  const int yi = q / G::A2, xi0 = 2 * (q - yi * G::A2), y = 1 + yi, z = 1 + (int)blockIdx.y;
  const int x0 = 2 * xi0 + ((y + z) & 1), o = (z * G::n + y) * G::P + xi0;
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (x0 + 2 * i >= 1 && x0 + 2 * i <= G::n - 2) u[(size_t)s * G::NS + o + i] = old[(size_t)s * G::BLK + o + i];
}

inline dim3 zmarch_grid(int n, int B, int* zslab) {
  const int slabs = apply_slabs(n, zslab);
  return dim3((unsigned)((n * n + 127) / 128), (unsigned)slabs, (unsigned)B);
}

// A node index that steps by the block size through a flat chunk of a sample: the index of its
// FP32 value (plain, or SPLIT: colour-split) without a division per node.
template <bool SPLIT>
struct FlatWalk {
  unsigned n, dq, dr, x, y, z, ns;
  __device__ __forceinline__ FlatWalk(int n_, unsigned i) {
    if (!SPLIT) return;
    n = (unsigned)n_;
    dq = kThreads / n;
    dr = kThreads - dq * n;
    z = i / (n * n);
    const unsigned rem = i - z * n * n;
    y = rem / n;
    x = rem - y * n;
  }
  __device__ __forceinline__ size_t at(unsigned i) const {
    return SPLIT ? (size_t)split_index((int)n, (int)x, (int)y, (int)z) : (size_t)i;
  }
  __device__ __forceinline__ void step() {
    if (!SPLIT) return;
    x += dr;
    y += dq;
    if (x >= n) {
      x -= n;
      ++y;
    }
    while (y >= n) {
      y -= n;
      ++z;
    }
  }
};

// The preconditioned residual z of a node: the FP32 correction of the V-cycle as it lies in the
// finest grid's iterate (MIX; SPLIT: in colour-split storage), or the FP64 one.
template <bool MIX, bool SPLIT>
struct PrecondZ {
  using Raw = typename std::conditional<MIX, float, double>::type;
  const void* z;
  __device__ __forceinline__ Raw raw(int n, int s, size_t n3, unsigned i, const FlatWalk<SPLIT>& w) const {
    return __ldg((const Raw*)z + (size_t)s * (SPLIT ? split_elems(n) : n3) + w.at(i));
  }
  __device__ __forceinline__ double at(int n, int s, size_t n3, unsigned i, const FlatWalk<SPLIT>& w) const {
    return widen(raw(n, s, n3, i, w));
  }
};

// r -= alpha q; r32 = (float) r for an FP32 preconditioner; partials of r.r and r.z (z: the
// previous preconditioned residual). The last block of a sample sums them and decides: the
// relative residual, the cycle count, whether the sample goes on (n_active) or is done with this
// iteration (fin, for k_cg_finish), and r.z (rzo). x is updated with p in k_p_update, which reads
// p anyway: 32 instead of 60 bytes per node here. Grid (NB, B).
template <bool MIX, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 4)
    k_cg_update(int n, const double* __restrict__ alpha, const double* __restrict__ q, double* __restrict__ r,
                PrecondZ<MIX, SPLIT> z, float* __restrict__ r32, double* part_rr, double* part_rz,
                double* __restrict__ rzo, const double* __restrict__ g2, double* __restrict__ relres,
                int* __restrict__ cycles, int* active, int* __restrict__ fin, double rtol, int max_cycles,
                int* __restrict__ n_active, int* tick) {
  const int s = blockIdx.y, NB = gridDim.x;
  if (!active[s]) {
    if (blockIdx.x == 0 && threadIdx.x == 0) fin[s] = 0;
    return;
  }
  const unsigned n3 = (unsigned)n * n * n;
  const unsigned chunk = (n3 + gridDim.x - 1) / gridDim.x;
  const unsigned lo = blockIdx.x * chunk, hi = lo + chunk < n3 ? lo + chunk : n3;
  const double a = alpha[s];
  double rr = 0.0, rz = 0.0;
  FlatWalk<SPLIT> w(n, lo + threadIdx.x);
  float* f = MIX ? r32 + (size_t)s * (SPLIT ? split_elems(n) : (size_t)n3) : nullptr;
  const double* qs = q + (size_t)s * n3;
  double* rs = r + (size_t)s * n3;
  // Two nodes a thread at a time, the next two loaded before these are computed: with four loaded
  // together every warp of the SM waited for memory at once and then queued at the FP64 pipe at once
  // (257^3 x 1: 152 -> 143 us a launch, x 2: 163 -> 149; the FP64 operations alone take 96 at x 1).
  struct Nodes {
    double q[2], r[2];
    typename PrecondZ<MIX, SPLIT>::Raw z[2];
    size_t f[2];
    unsigned i[2];
  };
  unsigned next = lo + threadIdx.x;
  auto fetch = [&](Nodes& v) {
#pragma unroll
    for (int k = 0; k < 2; ++k, next += kThreads) {
      const bool on = next < hi;
      v.i[k] = next;
      v.f[k] = w.at(next);
      v.q[k] = on ? qs[next] : 0.0;  // q vanishes on the boundary
      v.r[k] = on ? rs[next] : 0.0;
      v.z[k] = on ? z.raw(n, s, n3, next, w) : 0;
      w.step();
    }
  };
  auto use = [&](const Nodes& v) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      if (v.i[k] >= hi) break;
      const double rn = fma(-a, v.q[k], v.r[k]);
      rs[v.i[k]] = rn;
      if (MIX) f[v.f[k]] = (float)rn;
      rr = fma(rn, rn, rr);
      rz = fma(rn, widen(v.z[k]), rz);
    }
  };
  Nodes v0, v1;
  fetch(v0);
  while (v0.i[0] < hi) {
    fetch(v1);
    use(v0);
    if (v1.i[0] >= hi) break;
    fetch(v0);
    use(v1);
  }
  const double b1 = block_sum<kThreads>(rr);
  const double b2 = block_sum<kThreads>(rz);
  if (threadIdx.x == 0) {
    part_rr[(size_t)s * NB + blockIdx.x] = b1;
    part_rz[(size_t)s * NB + blockIdx.x] = b2;
  }
  if (last_block(tick + s, NB) && threadIdx.x < 32) {
    const double tz = warp_sum_fresh(part_rz + (size_t)s * NB, NB);
    const double tr = warp_sum_fresh(part_rr + (size_t)s * NB, NB);
    if (threadIdx.x == 0) {
      rzo[s] = tz;
      const double rel = g2[s] > 0.0 ? sqrt(tr / g2[s]) : 0.0;
      relres[s] = rel;
      const int c = cycles[s] + 1;
      cycles[s] = c;
      const int still = (rtol > 0.0) ? (rel > rtol && c < max_cycles) : (c < max_cycles);
      active[s] = still;
      fin[s] = !still;
      if (still) atomicAdd(n_active, 1);
    }
  }
}

// r.z of the new preconditioned residual z; the last block sets beta = (r.z - r.z_old) / rz (the
// flexible beta; not the first time) and rz = r.z. Grid (NB, B).
template <bool MIX, bool SPLIT>
__global__ void __launch_bounds__(kThreads, 8)
    k_precond_dot(int n, PrecondZ<MIX, SPLIT> z, const double* __restrict__ r, double* partial, int first,
                  const double* __restrict__ rzo, double* __restrict__ rz, double* __restrict__ beta, int* tick,
                  const int* __restrict__ active) {
  const int s = blockIdx.y, NB = gridDim.x;
  if (!active[s]) return;
  const unsigned n3 = (unsigned)n * n * n;
  const unsigned chunk = (n3 + gridDim.x - 1) / gridDim.x;
  const unsigned lo = blockIdx.x * chunk, hi = lo + chunk < n3 ? lo + chunk : n3;
  double acc = 0.0;
  const double* rs = r + (size_t)s * n3;
  FlatWalk<SPLIT> w(n, lo + threadIdx.x);
#pragma unroll 4
  for (unsigned i = lo + threadIdx.x; i < hi; i += kThreads) {
    acc = fma(rs[i], z.at(n, s, n3, i, w), acc);
    w.step();
  }
  const double b = block_sum<kThreads>(acc);
  if (threadIdx.x == 0) partial[(size_t)s * NB + blockIdx.x] = b;
  if (last_block(tick + s, NB) && threadIdx.x < 32) {
    const double t = warp_sum_fresh(partial + (size_t)s * NB, NB);
    if (threadIdx.x == 0) {
      if (!first) beta[s] = rz[s] != 0.0 ? (t - rzo[s]) / rz[s] : 0.0;
      rz[s] = t;
    }
  }
}

// The iteration's x += alpha p and the next direction p = z + beta p (first: p = z alone).
// Planes of active samples.
template <bool MIX, bool SPLIT>
__global__ void k_p_update(int n, int B, int first, const double* __restrict__ alpha, const double* __restrict__ beta,
                           const void* __restrict__ z, double* __restrict__ p, double* __restrict__ x,
                           const int* __restrict__ active) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // node of the plane
  if (q >= n * n) return;
  const int y = q / n, xx = q - y * n;
  const size_t n3 = (size_t)n * n * n;
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, zp = zz - s * n;
    if (!active[s]) continue;
    const size_t t = (size_t)s * n3 + (size_t)(zp * n * n + q);
    const double zv = MIX ? widen(((const float*)z)[SPLIT ? (size_t)s * split_elems(n) + split_index(n, xx, y, zp) : t])
                          : ((const double*)z)[t];
    if (first) {
      p[t] = zv;
    } else {
      const double pv = p[t];
      x[t] = fma(alpha[s], pv, x[t]);
      p[t] = fma(beta[s], pv, zv);
    }
  }
}

// x += alpha p of the samples that the iteration finished.
__global__ void k_cg_finish(int n, int B, const double* __restrict__ alpha, const double* __restrict__ p,
                            double* __restrict__ x, const int* __restrict__ fin) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // node of the plane
  if (q >= n * n) return;
  const size_t n3 = (size_t)n * n * n;
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, zp = zz - s * n;
    if (!fin[s]) continue;
    const size_t t = (size_t)s * n3 + (size_t)(zp * n * n + q);
    x[t] = fma(alpha[s], p[t], x[t]);
  }
}

__global__ void k_to_f32(size_t total, const double* __restrict__ a, float* __restrict__ b) {
  for (size_t t = (size_t)blockIdx.x * blockDim.x + threadIdx.x; t < total; t += (size_t)gridDim.x * blockDim.x)
    b[t] = (float)a[t];
}

// b = (float) a, a in the plain layout, b in colour-split storage (plane launch).
__global__ void k_to_f32_split(int n, int B, const double* __restrict__ a, float* __restrict__ b) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x;  // node of the plane
  if (q >= n * n) return;
  const int y = q / n, x = q - y * n;
  const size_t n3 = (size_t)n * n * n, ns = split_elems(n);
  for (int zz = blockIdx.y; zz < B * n; zz += gridDim.y) {
    const int s = zz / n, z = zz - s * n;
    b[(size_t)s * ns + split_index(n, x, y, z)] = (float)a[(size_t)s * n3 + (size_t)(z * n * n + q)];
  }
}

// ---------------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------------
template <typename T>
struct Level {
  int n = 0;
  size_t n3 = 0;
  T *Kx = nullptr, *Ky = nullptr, *Kz = nullptr, *D = nullptr, *Dinv = nullptr;
  T *u = nullptr, *g = nullptr, *r = nullptr;
  T* u2 = nullptr;  // spare iterate for the fused (double-buffered) sweep
  T* kn = nullptr;  // reciprocal nodal coefficient 1/k (FP32 grids: input of the nodal sweep)
};

template <typename T>
struct Hier {
  int L = 0, B = 0;
  Level<T> lv[kMaxLevels];
  double* Ainv = nullptr;
  // level-0 FP64 state
  double* g64 = nullptr;   // h^2 f
  double* D64 = nullptr;   // mixed: FP64 diagonal of the FP64 faces
  double *K64x = nullptr, *K64y = nullptr, *K64z = nullptr;  // mixed: FP64 faces of the finest grid
  int n_act = 0;           // host copy of the number of active samples (launch accounting)
  double* partial = nullptr;
  double* g2 = nullptr;
  double* relres = nullptr;
  int* cycles = nullptr;
  int* active = nullptr;
  int* n_active = nullptr;  // [2]: samples that go on, candidates to stop (k_norm_red)
  int* cand = nullptr;      // candidates to stop
  int* err = nullptr;  // device error word of bounded waits
  int NB = 1;   // partials per sample of the flat-chunk reductions (reduce_blocks)
  int NBu = 1;  // the same for k_cg_update (four blocks per SM)
  int NBz = 1;  // partials per sample of the column z-march kernels (apply_blocks)
  // flexible PCG (FP64 vectors on the finest grid) and per-sample scalars
  double *R = nullptr, *P = nullptr, *Q = nullptr, *Z = nullptr;
  double *part2 = nullptr, *rz = nullptr, *rzo = nullptr, *alpha = nullptr, *beta = nullptr;
  double* part_apply = nullptr;  // partials of p.q (k_apply_dot_z's partition)
  int* tick = nullptr;           // blocks of a sample that have finished (last_block)
  int tile[kMaxLevels] = {};      // fused-sweep tile shape per level
  bool fused[kMaxLevels] = {};    // fused (one pass) or two-pass smoother per level
  bool nodal[kMaxLevels] = {};    // two-pass sweep on the nodal coefficient (FP32)
  bool p1 = false;                // P1 finite elements: P1 transfers instead of FW / trilinear
  bool split = false;             // FP32 hierarchy in colour-split storage (MLMC_SMOOTH_SPLIT)
  bool tail_finest = false;       // the one-launch cycle may start on the finest grid (FMG)
  cudaError_t failed = cudaSuccess;  // a kernel of the cycle that could not be launched (GraphRunner reports it)
};

// Lays out the workspace. Level-0 u of FP64 solves is the caller's array (not carved).
template <typename T>
void layout(Hier<T>& H, Carver& c, int B, int n, bool mixed, bool cg) {
  H.B = B;
  H.L = hierarchy_depth(n);
  int nl = n;
  for (int j = 0; j < H.L; ++j) {
    Level<T>& v = H.lv[j];
    v.n = nl;
    v.n3 = cube(nl);
    const size_t e = (size_t)B * v.n3;
    // room for the colour-split storage (2 n^2 P instead of n^3 elements per sample, P =
    // (n + 1) / 2 rounded up to a multiple of 4) where a solve may take it: u, g, r and 1/k
    // of FP32 correction cycles; every array of FP64 stationary cycles (not of CG)
    const bool split64 = !mixed && !cg;
    const size_t es = (size_t)B * split_elems(nl);
    const size_t ef = split64 ? es : e, eu = (mixed || split64) ? es : e;
    v.Kx = c.template take<T>(ef);
    v.Ky = c.template take<T>(ef);
    v.Kz = c.template take<T>(ef);
    v.D = c.template take<T>(ef);
    v.Dinv = c.template take<T>(ef);
    // level 0 of an FP64 solve iterates in a copy of the caller's u (so that every array
    // the smoothers stage is carved here, with slack behind it); its g is g64 (or R for CG),
    // or the colour-split copy of g64 (MLMC_SMOOTH_SPLIT)
    v.u = c.template take<T>(eu);
    if (j > 0 || mixed || split64) v.g = c.template take<T>(eu);
    if (j < H.L - 1) v.u2 = c.template take<T>(e);
    if (j < H.L - 1) v.r = c.template take<T>(eu);
    if (mixed && j < H.L - 1) v.kn = c.template take<T>(es);
    nl = (nl + 1) / 2;
  }
  const size_t e0 = (size_t)B * cube(n);
  H.g64 = c.template take<double>(e0);
  if (mixed) {
    H.D64 = c.template take<double>(e0);
    H.K64x = c.template take<double>(e0);
    H.K64y = c.template take<double>(e0);
    H.K64z = c.template take<double>(e0);
  }
  H.Ainv = c.template take<double>((size_t)B * 729);
  H.NB = reduce_blocks(cube(n));
  H.NBu = reduce_blocks(cube(n), 4);
  H.NBz = apply_blocks(n);
  H.partial = c.template take<double>((size_t)B * (H.NB > H.NBz ? H.NB : H.NBz));
  H.g2 = c.template take<double>(B);
  H.relres = c.template take<double>(B);
  H.cycles = c.template take<int>(B);
  H.active = c.template take<int>(B);
  H.n_active = c.template take<int>(2);
  H.cand = c.template take<int>(B);
  H.err = c.template take<int>(1);
  if (cg) {
    H.R = c.template take<double>(e0);
    H.P = c.template take<double>(e0);
    H.Q = c.template take<double>(e0);
    if (mixed && n <= kCtaMaxN) H.Z = c.template take<double>(e0);  // the small-grid engine's
    H.tick = c.template take<int>(B);
    H.part2 = c.template take<double>((size_t)B * H.NB);
    H.part_apply = c.template take<double>((size_t)B * apply_blocks(n));
    H.rz = c.template take<double>(B);
    H.rzo = c.template take<double>(B);
    H.alpha = c.template take<double>(B);
    H.beta = c.template take<double>(B);
  }
}

template <typename T>
struct Names;
template <>
struct Names<double> {
  static constexpr const char* rbgs = "rbgs_f64";
  static constexpr const char* residual = "residual_f64";
  static constexpr const char* restrict_ = "restrict_f64";
  static constexpr const char* prolong = "prolong_f64";
  static constexpr const char* faces = "faces_f64";
  static constexpr const char* diag = "diag_f64";
  static constexpr const char* coarse = "coarse_apply_f64";
};
template <>
struct Names<float> {
  static constexpr const char* rbgs = "rbgs_f32";
  static constexpr const char* residual = "residual_f32";
  static constexpr const char* restrict_ = "restrict_f32";
  static constexpr const char* prolong = "prolong_f32";
  static constexpr const char* faces = "faces_f32";
  static constexpr const char* diag = "diag_f32";
  static constexpr const char* coarse = "coarse_apply_f32";
};

// groups of a colour row with an interior node, `nodes` values of x each (SplitGeo's A4, A2)
inline int split_groups(int n, int nodes) { return n > nodes + 1 ? (n - 1) / nodes : 1; }

inline double interior(int n) { return (double)(n - 2) * (n - 2) * (n - 2); }

// Red-black sweeps start on red and end on black, and a colour pass reads the other colour
// only. The V-cycle uses that three times: from a zero guess the first red pass is g / D
// (zero_pass: no product, and no clearing of u, whose boundary is zeroed once per solve);
// after a pre-smoothing sweep the black residuals are zero up to rounding, so the residual
// and the restriction take the red nodes alone; before a post-smoothing sweep the correction
// is interpolated to the black nodes alone (the red pass overwrites the red ones unread). An
// FP64 V(2,2) cycle on stored faces spends 28 + 3.5 + 1.7 + 1.6 FP64 operations per node on
// the finest grid instead of 28 + 7 + 3.4 + 2.75.
// Measured: FP64 solves of 65^3 x 19 10.42 -> 9.37 ms, the 129^3 / 65^3 level of 24 samples
// 83.5 -> 75.6 ms, the 17^3 level of 4096 samples (small-grid engine) 35.1 -> 32.7 ms, mixed
// refinement of 33^3 x 48 5.38 -> 4.81 ms, the mixed 257^3 / 129^3 level 43.9 -> 41.5 ms.
template <typename T>
inline bool zero_pass(const Hier<T>& H, int j, int nu1) {
  return j == H.L - 1 || (nu1 > 0 && !H.fused[j]);
}

// Cycle from a zero guess on grid j: clears u where the cycle's first pass reads it.
template <typename T>
cudaError_t clear_guess(const Hier<T>& H, int j, int nu1, cudaStream_t st) {
  if (zero_pass(H, j, nu1)) return cudaSuccess;
  const Level<T>& v = H.lv[j];
  return cudaMemsetAsync(v.u, 0, (size_t)H.B * (H.split ? split_elems(v.n) : v.n3) * sizeof(T), st);
}

// zero: u is zero on entry (cleared by clear_guess, where that is needed).
// red_done: the first red pass has been taken already (finest grid, k_rbgs_norm_split).
template <typename T>
void vcycle(Hier<T>& H, int j, int nu1, int nu2, cudaStream_t st, bool zero, bool red_done = false);

// ---------------------------------------------------------------------------------
// The V-cycle below a grid of at most 17^3 nodes as one launch, one block per sample.
// As launches its 20 (9^3: 10) passes are bound by launch latency, about 2.3 us each, for any
// batch up to a few hundred samples. Here the iterate, the right-hand side and the red residuals
// of every grid sit in shared memory (FP64: 112 KB from 17^3, two blocks per SM) and the passes
// are separated by block barriers; FP32 coefficients are staged too (nodal 1/k or stored faces),
// FP64 faces are read from L2 in the storage they have (plain or colour-split). Every node takes
// the batched kernels' operations in their order, so the iterates are theirs bit for bit. A red
// node (x, y, z) has an even linear index (N is odd), hence the half-size residual array. What
// bounds it: FP64 one SM's FP64 pipe (about 26 us a V(2,2) cycle from 17^3, whatever the batch up
// to two blocks an SM), FP32 the barriers. A mixed 33^3 x 48 solve 4.81 -> 3.81 ms (608 -> 256
// launches), an FP64 65^3 x 19 solve 9.03 -> 8.57, the 65^3 P1 / FMG level of 108 samples 21.9 ->
// 20.3, the 129^3 level of 24 66.0 -> 65.3; one launch takes 33 us (FP32, 2 samples) to 94 us
// (FP64 V(4,4), 108 samples).
// ---------------------------------------------------------------------------------
constexpr int kTailN = 17, kTailThreads = 512;
template <typename T>
struct TailLevel {
  const T *Kx, *Ky, *Kz, *D, *Dinv, *kn;  // kn: the nodal sweep of FP32 grids, else NULL
  const T* g;
  T* u;
};
template <typename T>
struct TailArgs {
  TailLevel<T> lv[2];  // from the finest grid of the tail (17^3 or 9^3)
  const double* Ainv;
  const int* active;
  int nu1, nu2, zero;
};

// One grid of the tail in a block: shared u, g, r and its coefficients (CS: colour-split FP64
// arrays in global memory; otherwise plain, shared for FP32 and global for FP64).
template <typename T, int N, bool CS>
struct TailGrid {
  T *u, *g, *r;
  const T *Kx, *Ky, *Kz, *D, *Dinv, *kn;
  static constexpr int N1 = N, N2 = N * N, N3 = N * N * N, M = N - 2, HALF = (N - 1) / 2;
  static constexpr int P = (((N + 1) / 2) + 3) & ~3, BLK = N * N * P;
  static constexpr int shared_iter = 2 * N3 + (N3 + 1) / 2;  // elements of u, g, r
  __device__ static __forceinline__ int at(int x, int y, int z) {
    return CS ? ((x + y + z) & 1) * BLK + (z * N + y) * P + (x >> 1) : (z * N + y) * N + x;
  }
  // node `it` of the colour, or false where the row has no such node
  __device__ static __forceinline__ bool node(int it, int colour, int& x, int& y, int& z) {
    const int zi = it / (M * HALF), q = it - zi * (M * HALF), yi = q / HALF;
    z = 1 + zi;
    y = 1 + yi;
    x = (((1 + y + z) & 1) == colour ? 1 : 2) + 2 * (q - yi * HALF);
    return x <= N - 2;
  }
  __device__ void pass(int colour, bool zero) const {
    for (int it = threadIdx.x; it < M * M * HALF; it += kTailThreads) {
      int x, y, z;
      if (!node(it, colour, x, y, z)) continue;
      const int p = (z * N + y) * N + x;
      if constexpr (sizeof(T) == 4) {
        if (kn) {
          u[p] = zero ? nodal_update<true>(kn[p], g[p], kn[p - 1], 0.f, kn[p + 1], 0.f, kn[p - N], 0.f, kn[p + N], 0.f,
                                           kn[p - N2], 0.f, kn[p + N2], 0.f)
                      : nodal_update(kn[p], g[p], kn[p - 1], u[p - 1], kn[p + 1], u[p + 1], kn[p - N], u[p - N],
                                     kn[p + N], u[p + N], kn[p - N2], u[p - N2], kn[p + N2], u[p + N2]);
          continue;
        }
      }
      const int o = at(x, y, z);
      T acc = g[p];
      if (!zero) {
        acc = fma(Kx[at(x - 1, y, z)], u[p - 1], acc);
        acc = fma(Kx[o], u[p + 1], acc);
        acc = fma(Ky[at(x, y - 1, z)], u[p - N], acc);
        acc = fma(Ky[o], u[p + N], acc);
        acc = fma(Kz[at(x, y, z - 1)], u[p - N2], acc);
        acc = fma(Kz[o], u[p + N2], acc);
      }
      u[p] = acc * Dinv[o];
    }
    __syncthreads();
  }
  __device__ void red_residual() const {
    for (int it = threadIdx.x; it < M * M * HALF; it += kTailThreads) {
      int x, y, z;
      if (!node(it, 0, x, y, z)) continue;
      const int p = (z * N + y) * N + x;
      if constexpr (sizeof(T) == 4) {
        if (kn) {
          r[p >> 1] = nodal_residual(kn[p], g[p], u[p], kn[p - 1], u[p - 1], kn[p + 1], u[p + 1], kn[p - N], u[p - N],
                                     kn[p + N], u[p + N], kn[p - N2], u[p - N2], kn[p + N2], u[p + N2]);
          continue;
        }
      }
      const int o = at(x, y, z);
      T rr = fma(-D[o], u[p], g[p]);
      rr = fma(Kx[at(x - 1, y, z)], u[p - 1], rr);
      rr = fma(Kx[o], u[p + 1], rr);
      rr = fma(Ky[at(x, y - 1, z)], u[p - N], rr);
      rr = fma(Ky[o], u[p + N], rr);
      rr = fma(Kz[at(x, y, z - 1)], u[p - N2], rr);
      rr = fma(Kz[o], u[p + N2], rr);
      r[p >> 1] = rr;
    }
    __syncthreads();
  }
  // g of the coarse grid from the red residuals (k_restrict_red, P1: k_restrict_p1_red)
  template <bool P1>
  __device__ void restrict_to(T* gc) const {
    constexpr int NC = (N + 1) / 2, MC = NC - 2;
    for (int it = threadIdx.x; it < MC * MC * MC; it += kTailThreads) {
      const int Z = 1 + it / (MC * MC), q = it % (MC * MC), Y = 1 + q / MC, X = 1 + q % MC;
      const int p = (2 * Z * N + 2 * Y) * N + 2 * X;
      auto R = [&](int dx, int dy, int dz) { return r[(p + (dz * N + dy) * N + dx) >> 1]; };
      T v = 0;
      if (P1) {
        T acc = R(-1, -1, 0) + R(1, 1, 0);
        acc += R(0, -1, -1) + R(0, 1, 1);
        acc += R(-1, 0, -1) + R(1, 0, 1);
        v = T(0.5) * R(0, 0, 0) + T(0.25) * acc;
      } else {
#pragma unroll
        for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
          for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
            for (int dx = -1; dx <= 1; ++dx) {
              if ((dx + dy + dz) & 1) continue;
              const T wgt = (T)((2 - abs(dx)) * (2 - abs(dy)) * (2 - abs(dz))) * (T)(1.0 / 16.0);
              v = fma(wgt, R(dx, dy, dz), v);
            }
      }
      gc[(Z * NC + Y) * NC + X] = v;
    }
    __syncthreads();
  }
  // u += the interpolated coarse correction at the black nodes (k_prolong_blk, k_prolong_p1_black)
  template <bool P1>
  __device__ void prolong_from(const T* ec) const {
    constexpr int NC = (N + 1) / 2, MC = NC - 1;
    if (P1) {
      for (int it = threadIdx.x; it < M * M * HALF; it += kTailThreads) {
        int x, y, z;
        if (!node(it, 1, x, y, z)) continue;
        const int dx = x & 1, dy = y & 1, dz = z & 1, c = ((z >> 1) * NC + (y >> 1)) * NC + (x >> 1);
        u[(z * N + y) * N + x] += T(0.5) * (ec[c] + ec[c + (dz * NC + dy) * NC + dx]);
      }
    } else {
      for (int it = threadIdx.x; it < MC * MC * MC; it += kTailThreads) {
        const int Z = it / (MC * MC), q = it % (MC * MC), Y = q / MC, X = q % MC;
        const T* e = ec + (Z * NC + Y) * NC + X;
        const T c[8] = {e[0], e[1], e[NC], e[NC + 1], e[NC * NC], e[NC * NC + 1], e[NC * NC + NC], e[NC * NC + NC + 1]};
        T v[8];
        prolong_block_sums(c, v);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int dx = k & 1, dy = (k >> 1) & 1, dz = k >> 2;
          if (!((dx + dy + dz) & 1)) continue;
          const int x = 2 * X + dx, y = 2 * Y + dy, z = 2 * Z + dz;
          if (x < 1 || y < 1 || z < 1 || x > N - 2 || y > N - 2 || z > N - 2) continue;
          const T w = dx + dy + dz == 1 ? T(0.5) : T(0.125);
          u[(z * N + y) * N + x] += w * v[k];
        }
      }
    }
    __syncthreads();
  }
};

// FP32 coefficients staged in shared memory: nodal 1/k, or Kx, Ky, Kz, D, 1/D
inline int tail_coef_arrays(bool f32, bool nodal) { return f32 ? (nodal ? 1 : 5) : 0; }

template <typename T, int N0, bool SPLIT, bool P1>
__global__ void __launch_bounds__(kTailThreads) k_vcycle_tail(TailArgs<T> A) {
  constexpr bool F32 = sizeof(T) == 4, CS = SPLIT && !F32;
  constexpr int LV = N0 == 17 ? 2 : 1;
  using G0 = TailGrid<T, N0, CS>;
  using G1 = TailGrid<T, 9, CS>;
  extern __shared__ __align__(16) unsigned char tail_smem[];
  const int s = blockIdx.x, tid = threadIdx.x;
  if (!A.active[s]) return;
  T* sm = reinterpret_cast<T*>(tail_smem);
  T* const base = sm;
  G0 a;
  G1 b;
  auto carve = [&](auto& G) {
    using G_ = typename std::remove_reference<decltype(G)>::type;
    G.u = sm;
    G.g = sm + G_::N3;
    G.r = sm + 2 * G_::N3;
    sm += G_::shared_iter;
  };
  carve(a);
  if (LV == 2) carve(b);
  T* const u5 = sm;
  T* const g5 = sm + 125;
  sm += 250;
  for (int i = tid; i < (int)(sm - base); i += kTailThreads) base[i] = T(0);
  // the coefficients: plain FP32 copies in shared memory, FP64 where they are
  auto coefs = [&](auto& G, const TailLevel<T>& L) {
    using G_ = typename std::remove_reference<decltype(G)>::type;
    constexpr size_t NS = SPLIT ? (size_t)2 * G_::BLK : (size_t)G_::N3;
    const size_t o = (size_t)s * NS;
    G.kn = nullptr;
    if constexpr (!F32) {
      G.Kx = L.Kx + o;
      G.Ky = L.Ky + o;
      G.Kz = L.Kz + o;
      G.D = L.D + o;
      G.Dinv = L.Dinv + o;
    } else {
      auto stage = [&](const T* src) -> const T* {
        T* dst = sm;
        for (int i = tid; i < G_::N3; i += kTailThreads) {
          const int z = i / G_::N2, q = i - z * G_::N2, y = q / G_::N1, x = q - y * G_::N1;
          dst[i] = src[o + (SPLIT ? ((x + y + z) & 1) * G_::BLK + (z * G_::N1 + y) * G_::P + (x >> 1) : i)];
        }
        sm += G_::N3;
        return dst;
      };
      if (L.kn) {
        G.kn = stage(L.kn);
      } else {
        G.Kx = stage(L.Kx);
        G.Ky = stage(L.Ky);
        G.Kz = stage(L.Kz);
        G.D = stage(L.D);
        G.Dinv = stage(L.Dinv);
      }
    }
  };
  coefs(a, A.lv[0]);
  if (LV == 2) coefs(b, A.lv[1]);
  __syncthreads();
  // interior nodes of the finest grid of the tail: its g and, from a non-zero guess, its u
  auto each = [&](auto fn) {
    constexpr int M = N0 - 2;
    for (int i = tid; i < M * M * M; i += kTailThreads) {
      const int z = 1 + i / (M * M), q = i % (M * M), y = 1 + q / M, x = 1 + q % M;
      const size_t o = SPLIT ? (size_t)s * 2 * G0::BLK + (size_t)(((x + y + z) & 1) * G0::BLK + (z * N0 + y) * G0::P + (x >> 1))
                             : (size_t)s * G0::N3 + (size_t)((z * N0 + y) * N0 + x);
      fn((z * N0 + y) * N0 + x, o);
    }
  };
  each([&](int p, size_t o) {
    a.g[p] = A.lv[0].g[o];
    if (!A.zero) a.u[p] = A.lv[0].u[o];
  });
  __syncthreads();
  auto down = [&](auto& G, T* gc, bool zero) {
    for (int k = 0; k < A.nu1; ++k)
      for (int c = 0; c < 2; ++c) G.pass(c, zero && k == 0 && c == 0);
    G.red_residual();
    G.template restrict_to<P1>(gc);
  };
  auto up = [&](auto& G, const T* ec) {
    G.template prolong_from<P1>(ec);
    for (int k = 0; k < A.nu2; ++k)
      for (int c = 0; c < 2; ++c) G.pass(c, false);
  };
  down(a, LV == 2 ? b.g : g5, A.zero != 0);
  if constexpr (LV == 2) down(b, g5, true);
  if (tid < 27) {  // the exact solve (k_coarse_apply)
    const double* X = A.Ainv + (size_t)s * 729 + (size_t)tid * 27;
    double v = 0.0;
    for (int q = 0; q < 27; ++q)
      v = fma(X[q], (double)g5[((1 + q / 9) * 5 + 1 + (q / 3) % 3) * 5 + 1 + q % 3], v);
    u5[((1 + tid / 9) * 5 + 1 + (tid / 3) % 3) * 5 + 1 + tid % 3] = (T)v;
  }
  __syncthreads();
  if constexpr (LV == 2) up(b, u5);
  up(a, LV == 2 ? b.u : u5);
  each([&](int p, size_t o) { A.lv[0].u[o] = a.u[p]; });
}

// Whether the cycle from grid j down runs as one launch: grids of 17^3 or 9^3 below the finest
// (for an FMG cycle, which has no small-grid engine, also the finest grid, unless the batched
// engine is asked for), with both pre- and post-smoothing (the red-black shortcuts).
template <typename T>
inline bool tail_applies(const Hier<T>& H, int j, int nu1, int nu2) {
  const int n = H.lv[j].n;
  return (n == 17 || n == 9) && (j > 0 || H.tail_finest) && nu1 > 0 && nu2 > 0;
}

template <typename T, int N0, bool SPLIT, bool P1>
cudaError_t tail_launch(const TailArgs<T>& A, int B, int coef0, int coef1, double nodes, cudaStream_t st) {
  constexpr int N1 = 9;
  const size_t elems = (size_t)TailGrid<T, N0, false>::shared_iter + 250 + (size_t)coef0 * N0 * N0 * N0 +
                       (N0 == 17 ? (size_t)TailGrid<T, N1, false>::shared_iter + (size_t)coef1 * N1 * N1 * N1 : 0);
  const cudaError_t attr = allow_dynamic_smem<k_vcycle_tail<T, N0, SPLIT, P1>>(200 * 1024);
  if (attr != cudaSuccess) return attr;
  const int nu = A.nu1 + A.nu2;
  MLMC_LAUNCH(prof::sized(sizeof(T) == 8 ? "vcycle_tail_f64" : "vcycle_tail_f32", N0),
              nodes * nu * 7.0 * (double)sizeof(T), nodes * (nu * 13.0 + 14.0), st,
              (k_vcycle_tail<T, N0, SPLIT, P1><<<B, kTailThreads, elems * sizeof(T), st>>>(A)));
  return cudaSuccess;
}

template <typename T>
void vcycle_tail(Hier<T>& H, int j, int nu1, int nu2, cudaStream_t st, bool zero) {
  TailArgs<T> A{};
  const int n = H.lv[j].n, B = H.B;
  int coef[2] = {0, 0};
  for (int k = 0; k < (n == 17 ? 2 : 1); ++k) {
    const Level<T>& v = H.lv[j + k];
    const bool nodal = sizeof(T) == 4 && (H.split || H.nodal[j + k]);
    A.lv[k] = {v.Kx, v.Ky, v.Kz, v.D, v.Dinv, nodal ? v.kn : nullptr, v.g, v.u};
    coef[k] = tail_coef_arrays(sizeof(T) == 4, nodal);
  }
  A.Ainv = H.Ainv;
  A.active = H.active;
  A.nu1 = nu1;
  A.nu2 = nu2;
  A.zero = zero ? 1 : 0;
  const double nodes = (double)H.n_act * interior(n) * 8.0 / 7.0;
  auto go = [&](auto n0) {
    constexpr int N0 = decltype(n0)::value;
    if constexpr (sizeof(T) == 8) {
      if (H.split && H.p1) return tail_launch<T, N0, true, true>(A, B, 0, 0, nodes, st);
      if (H.split) return tail_launch<T, N0, true, false>(A, B, 0, 0, nodes, st);
      if (H.p1) return tail_launch<T, N0, false, true>(A, B, 0, 0, nodes, st);
      return tail_launch<T, N0, false, false>(A, B, 0, 0, nodes, st);
    } else {
      if (H.split) return tail_launch<T, N0, true, false>(A, B, coef[0], coef[1], nodes, st);
      return tail_launch<T, N0, false, false>(A, B, coef[0], coef[1], nodes, st);
    }
  };
  const cudaError_t e = n == 17 ? go(std::integral_constant<int, 17>()) : go(std::integral_constant<int, 9>());
  if (e != cudaSuccess) H.failed = e;
}

// One level of the V-cycle on colour-split FP32 storage: nodal-coefficient colour passes,
// the residual into the plain r, full weighting into the coarse grid's split g, the
// coarser levels, the trilinear correction on split storage, post-smoothing.
template <typename T>
void vcycle_split(Hier<T>& H, int j, int nu1, int nu2, cudaStream_t st, bool zero) {
  Level<T>& v = H.lv[j];
  Level<T>& w = H.lv[j + 1];
  const int* act = H.active;
  const int B = H.B, m = v.n - 2;
  const double Ba = (double)H.n_act, W = 4.0;
  float* u = (float*)(void*)v.u;
  const float* g = (const float*)(const void*)v.g;
  const float* kn = (const float*)(const void*)v.kn;
  const dim3 gs((unsigned)((m * split_groups(v.n, 8) + 127) / 128), (unsigned)m, (unsigned)B);
  auto smooth = [&](int sweeps, bool from_zero) {
    for (int s = 0; s < sweeps; ++s)
      for (int c = 0; c < 2; ++c) {
        if (from_zero && s == 0 && c == 0)
          MLMC_LAUNCH(prof::sized("rbgs_split_f32", v.n), Ba * interior(v.n) * 1.5 * W, Ba * interior(v.n) * 0.5 * 25.0,
                      st, MLMC_SPLIT_DISPATCH(v.n, (k_rbgs_split<LG, true><<<gs, 128, 0, st>>>(c, kn, g, u, act))));
        else
          MLMC_LAUNCH(prof::sized("rbgs_split_f32", v.n), Ba * interior(v.n) * 2.0 * W, Ba * interior(v.n) * 0.5 * 37.0,
                      st, MLMC_SPLIT_DISPATCH(v.n, (k_rbgs_split<LG><<<gs, 128, 0, st>>>(c, kn, g, u, act))));
      }
  };
  smooth(nu1, zero);
  const unsigned groups = (unsigned)((m * split_groups(v.n, 8) + 127) / 128);
  float* r = (float*)(void*)v.r;  // colour-split r~ (room for n^2 (n+1) elements: carved as n^3 + slack)
  const dim3 rg((unsigned)(((w.n - 2) * (w.n - 2) + 127) / 128), (unsigned)(w.n - 2), (unsigned)B);
  if (nu1 > 0) {
    MLMC_LAUNCH(prof::sized("residual_split_f32", v.n), Ba * interior(v.n) * 3.0 * W, Ba * interior(v.n) * 18.5, st,
                MLMC_SPLIT_DISPATCH(v.n, (k_residual_split<LG, true><<<dim3(groups, (unsigned)m, (unsigned)B), 128, 0,
                                                                        st>>>(kn, g, u, r, act))));
    MLMC_LAUNCH(Names<T>::restrict_, Ba * (0.5 * (double)v.n3 + (double)w.n3) * W, Ba * interior(w.n) * 26.0, st,
                MLMC_SPLIT_DISPATCH(v.n, (k_restrict_split<LG, float, true><<<rg, 128, 0, st>>>(
                                             r, (float*)(void*)w.g, act))));
  } else {
    MLMC_LAUNCH(prof::sized("residual_split_f32", v.n), Ba * interior(v.n) * 4.0 * W, Ba * interior(v.n) * 37.0, st,
                MLMC_SPLIT_DISPATCH(v.n, (k_residual_split<LG><<<dim3(groups, (unsigned)(2 * m), (unsigned)B), 128, 0,
                                                                  st>>>(kn, g, u, r, act))));
    MLMC_LAUNCH(Names<T>::restrict_, Ba * ((double)v.n3 + (double)w.n3) * W, Ba * interior(w.n) * 54.0, st,
                MLMC_SPLIT_DISPATCH(v.n, (k_restrict_split<LG><<<rg, 128, 0, st>>>(r, (float*)(void*)w.g, act))));
  }
  clear_guess(H, j + 1, nu1, st);
  vcycle(H, j + 1, nu1, nu2, st, true);
  if (nu2 > 0)
    MLMC_LAUNCH(prof::sized("prolong_split_f32", v.n), Ba * ((double)v.n3 + (double)w.n3) * W,
                Ba * interior(v.n) * 2.2, st,
                MLMC_SPLIT_DISPATCH(v.n, (k_prolong_split<LG, true><<<dim3(groups, (unsigned)m, (unsigned)B), 128, 0,
                                                                       st>>>((const float*)(const void*)w.u, u,
                                                                             act))));
  else
    MLMC_LAUNCH(prof::sized("prolong_split_f32", v.n), Ba * (2.0 * (double)v.n3 + (double)w.n3) * W,
                Ba * interior(v.n) * 4.375, st,
                MLMC_SPLIT_DISPATCH(v.n, (k_prolong_split<LG><<<dim3(groups, (unsigned)m, (unsigned)(2 * B)), 128, 0,
                                                                 st>>>((const float*)(const void*)w.u, u, act))));
  smooth(nu2, false);
}

// u_j += the interpolation of grid j + 1's u (P1 or trilinear; plain or, for FP64, split
// storage). black: at the black nodes only (a red pass follows).
template <typename T>
void prolong_level(Hier<T>& H, int j, bool black, cudaStream_t st) {
  const Level<T>& v = H.lv[j];
  const Level<T>& w = H.lv[j + 1];
  const int* act = H.active;
  const int B = H.B, m = v.n - 2, mc = w.n - 1;
  const double Ba = (double)H.n_act, W = (double)sizeof(T);
  const double bytes = Ba * ((black ? 1.0 : 2.0) * (double)v.n3 + (double)w.n3) * W;
  if (H.p1) {
    const dim3 all = plane_grid(m * m, (long long)B * m), blk = plane_grid(m * mc, (long long)B * m);
    const double flops = Ba * interior(v.n) * (black ? 0.75 : 1.5);
    if (H.split && black)
      MLMC_LAUNCH("prolong_p1", bytes, flops, st,
                  (k_prolong_p1_black<T, true><<<blk, kPlaneThreads, 0, st>>>(v.n, B, w.u, v.u, act)));
    else if (H.split)
      MLMC_LAUNCH("prolong_p1", bytes, flops, st,
                  (k_prolong_p1<T, true><<<all, kPlaneThreads, 0, st>>>(v.n, B, w.u, v.u, act)));
    else if (black)
      MLMC_LAUNCH("prolong_p1", bytes, flops, st,
                  (k_prolong_p1_black<T, false><<<blk, kPlaneThreads, 0, st>>>(v.n, B, w.u, v.u, act)));
    else
      MLMC_LAUNCH("prolong_p1", bytes, flops, st,
                  (k_prolong_p1<T><<<all, kPlaneThreads, 0, st>>>(v.n, B, w.u, v.u, act)));
    return;
  }
  const double flops = Ba * interior(v.n) * (black ? 1.6 : 2.75);
  if (H.split) {
    if constexpr (sizeof(T) == 8) {
      const dim3 g((unsigned)((mc * mc + 127) / 128), (unsigned)mc, (unsigned)B);
      if (black)
        MLMC_LAUNCH(prof::sized("prolong_split_f64", v.n), bytes, flops, st,
                    MLMC_SPLIT_DISPATCH(v.n, (k_prolong_blk_split<LG, T, true><<<g, 128, 0, st>>>(w.u, v.u, act))));
      else
        MLMC_LAUNCH(prof::sized("prolong_split_f64", v.n), bytes, flops, st,
                    MLMC_SPLIT_DISPATCH(v.n, (k_prolong_blk_split<LG, T><<<g, 128, 0, st>>>(w.u, v.u, act))));
    }
    return;
  }
  const dim3 g = plane_grid(mc * mc, (long long)B * mc);
  if (black)
    MLMC_LAUNCH(Names<T>::prolong, bytes, flops, st,
                (k_prolong_blk<T, true><<<g, 128, 0, st>>>(v.n, B, w.u, v.u, act)));
  else
    MLMC_LAUNCH(Names<T>::prolong, bytes, flops, st, (k_prolong_blk<T><<<g, 128, 0, st>>>(v.n, B, w.u, v.u, act)));
}

// One level of the V-cycle on colour-split FP64 storage (stored faces): two-pass colour
// sweeps, the residual into split r, full weighting into the coarse split g, the coarser
// levels, the trilinear correction on split storage, post-smoothing.
template <typename T>
void vcycle_split64(Hier<T>& H, int j, int nu1, int nu2, cudaStream_t st, bool zero, bool red_done) {
  Level<T>& v = H.lv[j];
  Level<T>& w = H.lv[j + 1];
  const int* act = H.active;
  const int B = H.B, m = v.n - 2;
  const double Ba = (double)H.n_act, W = 8.0;
  const double* Kx = (const double*)(const void*)v.Kx;
  const double* Ky = (const double*)(const void*)v.Ky;
  const double* Kz = (const double*)(const void*)v.Kz;
  const double* D = (const double*)(const void*)v.D;
  const double* Dinv = (const double*)(const void*)v.Dinv;
  const double* g = (const double*)(const void*)v.g;
  double* u = (double*)(void*)v.u;
  double* r = (double*)(void*)v.r;
  const unsigned pairs = (unsigned)((m * split_groups(v.n, 4) + 127) / 128);
  const dim3 gs(pairs, (unsigned)m, (unsigned)B);
  auto smooth = [&](int sweeps, bool from_zero, bool skip_red) {
    for (int s = 0; s < sweeps; ++s)
      for (int c = 0; c < 2; ++c) {
        if (skip_red && s == 0 && c == 0) continue;
        if (from_zero && s == 0 && c == 0)
          MLMC_LAUNCH(prof::sized("rbgs_split_f64", v.n), Ba * interior(v.n) * 1.5 * W, Ba * interior(v.n) * 0.5, st,
                      MLMC_SPLIT_DISPATCH(v.n, (k_rbgs_split64<LG, true><<<gs, 128, 0, st>>>(c, Kx, Ky, Kz, Dinv, g, u,
                                                                                           act))));
        else
          MLMC_LAUNCH(prof::sized("rbgs_split_f64", v.n), Ba * interior(v.n) * 3.5 * W, Ba * interior(v.n) * 0.5 * 13.0,
                      st, MLMC_SPLIT_DISPATCH(v.n, (k_rbgs_split64<LG><<<gs, 128, 0, st>>>(c, Kx, Ky, Kz, Dinv, g, u,
                                                                                         act))));
      }
  };
  smooth(nu1, zero, red_done);
  const bool red = nu1 > 0, black = nu2 > 0;
  double* gc = (double*)(void*)w.g;
  if (red)
    MLMC_LAUNCH(prof::sized("residual_split_f64", v.n), Ba * interior(v.n) * 4.0 * W, Ba * interior(v.n) * 7.0, st,
                MLMC_SPLIT_DISPATCH(v.n, (k_residual_split64<LG, true><<<gs, 128, 0, st>>>(Kx, Ky, Kz, D, g, u, r,
                                                                                         act))));
  else
    MLMC_LAUNCH(prof::sized("residual_split_f64", v.n), Ba * interior(v.n) * 7.0 * W, Ba * interior(v.n) * 14.0, st,
                MLMC_SPLIT_DISPATCH(v.n, (k_residual_split64<LG><<<dim3(pairs, (unsigned)(2 * m), (unsigned)B), 128, 0,
                                                                    st>>>(Kx, Ky, Kz, D, g, u, r, act))));
  const dim3 rg((unsigned)(((w.n - 2) * (w.n - 2) + 127) / 128), (unsigned)(w.n - 2), (unsigned)B);
  const dim3 p1r = plane_grid((w.n - 2) * (w.n - 2), (long long)B * (w.n - 2));
  const double rbytes = Ba * ((red ? 0.5 : 1.0) * (double)v.n3 + (double)w.n3) * W;
  if (H.p1 && red)
    MLMC_LAUNCH("restrict_p1", rbytes, Ba * interior(w.n) * 8.0, st,
                (k_restrict_p1_red<double, true><<<p1r, kPlaneThreads, 0, st>>>(v.n, B, r, gc, act)));
  else if (H.p1)
    MLMC_LAUNCH("restrict_p1", rbytes, Ba * interior(w.n) * 16.0, st,
                (k_restrict_p1<double, true><<<p1r, kPlaneThreads, 0, st>>>(v.n, B, r, gc, act)));
  else if (red)
    MLMC_LAUNCH(Names<T>::restrict_, rbytes, Ba * interior(w.n) * 26.0, st,
                MLMC_SPLIT_DISPATCH(v.n, (k_restrict_split<LG, double, true><<<rg, 128, 0, st>>>(r, gc, act))));
  else
    MLMC_LAUNCH(Names<T>::restrict_, rbytes, Ba * interior(w.n) * 54.0, st,
                MLMC_SPLIT_DISPATCH(v.n, (k_restrict_split<LG, double><<<rg, 128, 0, st>>>(r, gc, act))));
  clear_guess(H, j + 1, nu1, st);
  vcycle(H, j + 1, nu1, nu2, st, true);
  prolong_level(H, j, black, st);
  smooth(nu2, false, false);
}

template <typename T>
void vcycle(Hier<T>& H, int j, int nu1, int nu2, cudaStream_t st, bool zero, bool red_done) {
  Level<T>& v = H.lv[j];
  const int* act = H.active;
  const int B = H.B;
  // launches cover all B samples; masked (finished) samples do no work, so the
  // algorithmic bytes and flops count the active ones only
  const double Ba = (double)H.n_act;
  const double W = (double)sizeof(T);
  if (j == H.L - 1) {
    if (H.split)
      MLMC_LAUNCH(Names<T>::coarse, Ba * (729.0 * 8 + 54 * W), Ba * 27 * 54.0, st,
                  (k_coarse_apply<T, true><<<(B * 27 + 127) / 128, 128, 0, st>>>(B, H.Ainv, v.g, v.u, act)));
    else
      MLMC_LAUNCH(Names<T>::coarse, Ba * (729.0 * 8 + 54 * W), Ba * 27 * 54.0, st,
                  (k_coarse_apply<T><<<(B * 27 + 127) / 128, 128, 0, st>>>(B, H.Ainv, v.g, v.u, act)));
    return;
  }
  if (tail_applies(H, j, nu1, nu2)) {
    vcycle_tail(H, j, nu1, nu2, st, zero);
    return;
  }
  if (H.split) {
    if constexpr (sizeof(T) == 4)
      vcycle_split(H, j, nu1, nu2, st, zero);
    else
      vcycle_split64(H, j, nu1, nu2, st, zero, red_done);
    return;
  }
  const int m = v.n - 2;
  const dim3 gs = plane_grid(m * ((v.n - 1) / 2), (long long)B * m);
  // one colour: half of the 7 words per node of a full sweep; 13 flops per updated node
  const double sweep_bytes = Ba * interior(v.n) * 3.5 * W, sweep_flops = Ba * interior(v.n) * 0.5 * 13.0;
  auto smooth = [&](int sweeps, bool from_zero) {
    for (int s = 0; s < sweeps; ++s) {
      const bool z0 = from_zero && s == 0 && !H.fused[j];
      if (z0 && !H.nodal[j])
        MLMC_LAUNCH(prof::sized(Names<T>::rbgs, v.n), Ba * interior(v.n) * 1.5 * W, Ba * interior(v.n) * 0.5, st,
                    (k_rbgs<T, true><<<gs, kPlaneThreads, 0, st>>>(0, v.n, B, v.Kx, v.Ky, v.Kz, v.Dinv, v.g, v.u, act)));
      if constexpr (sizeof(T) == 4) {
        if (H.nodal[j]) {
          const float* kn = (const float*)v.kn;
          const float* g = (const float*)v.g;
          float* u = (float*)v.u;
          if (z0)
            MLMC_LAUNCH(prof::sized("rbgs_nodal_f32", v.n), Ba * interior(v.n) * 1.5 * W,
                        Ba * interior(v.n) * 0.5 * 25.0, st,
                        (k_rbgs_nodal<true><<<gs, kPlaneThreads, 0, st>>>(0, v.n, B, kn, g, u, act)));
          for (int c = z0 ? 1 : 0; c < 2; ++c)
            MLMC_LAUNCH(prof::sized("rbgs_nodal_f32", v.n), Ba * interior(v.n) * 2.0 * W, Ba * interior(v.n) * 0.5 * 37.0, st,
                        (k_rbgs_nodal<false><<<gs, kPlaneThreads, 0, st>>>(c, v.n, B, kn, g, u, act)));
          continue;
        }
      }
      if (H.fused[j]) {
        rbgs_fused_sweep<T>(H.tile[j], v.n, B, v.Kx, v.Ky, v.Kz, v.Dinv, v.g, v.u, v.u2, act, H.err, st, Ba);
        T* t = v.u;
        v.u = v.u2;
        v.u2 = t;
      } else {
        for (int c = z0 ? 1 : 0; c < 2; ++c)
          MLMC_LAUNCH(prof::sized(Names<T>::rbgs, v.n), sweep_bytes, sweep_flops, st,
                      (k_rbgs<T><<<gs, kPlaneThreads, 0, st>>>(c, v.n, B, v.Kx, v.Ky, v.Kz, v.Dinv, v.g, v.u, act)));
      }
    }
  };
  smooth(nu1, zero);
  const bool red = nu1 > 0;
  bool nodal_res = false;
  if constexpr (sizeof(T) == 4) {
    if (H.nodal[j]) {
      const float* kn = (const float*)v.kn;
      const float* g = (const float*)v.g;
      const float* u = (const float*)v.u;
      if (red)
        MLMC_LAUNCH(prof::sized("residual_nodal_f32", v.n), Ba * interior(v.n) * 3.0 * W, Ba * interior(v.n) * 18.5, st,
                    (k_residual_nodal<true><<<plane_grid(v.n * ((v.n + 1) / 2), (long long)B * v.n), kPlaneThreads, 0,
                                              st>>>(v.n, B, kn, g, u, (float*)v.r, act)));
      else
        MLMC_LAUNCH(prof::sized("residual_nodal_f32", v.n), Ba * interior(v.n) * 4.0 * W, Ba * interior(v.n) * 37.0, st,
                    (k_residual_nodal<false><<<plane_grid(v.n * v.n, (long long)B * v.n), kPlaneThreads, 0, st>>>(
                        v.n, B, kn, g, u, (float*)v.r, act)));
      nodal_res = true;
    }
  }
  if (!nodal_res && red) {
    MLMC_LAUNCH(prof::sized(Names<T>::residual, v.n), Ba * interior(v.n) * 4.0 * W, Ba * interior(v.n) * 7.0, st,
                (k_residual_red<T><<<gs, kPlaneThreads, 0, st>>>(v.n, B, v.Kx, v.Ky, v.Kz, v.D, v.g, v.u, v.r, act)));
  } else if (!nodal_res) {
    int zs = 0;
    const dim3 rz = zmarch_grid(v.n, B, &zs);
    MLMC_LAUNCH(prof::sized(Names<T>::residual, v.n), Ba * interior(v.n) * 7.0 * W, Ba * interior(v.n) * 14.0, st,
                (k_residual_z<T, T, T, T><<<rz, 128, 0, st>>>(v.n, zs, v.Kx, v.Ky, v.Kz, v.D, v.g, v.u, v.r, nullptr,
                                                              act)));
  }
  Level<T>& w = H.lv[j + 1];
  const dim3 p1r = plane_grid((w.n - 2) * (w.n - 2), (long long)B * (w.n - 2));
  const dim3 fwr = plane_grid((w.n - 2) * (w.n - 1), (long long)B * (w.n - 2));
  const double rbytes = Ba * ((red ? 0.5 : 1.0) * (double)v.n3 + (double)w.n3) * W;
  if (H.p1 && red)
    MLMC_LAUNCH("restrict_p1", rbytes, Ba * interior(w.n) * 8.0, st,
                (k_restrict_p1_red<T, false><<<p1r, kPlaneThreads, 0, st>>>(v.n, B, v.r, w.g, act)));
  else if (H.p1)
    MLMC_LAUNCH("restrict_p1", rbytes, Ba * interior(w.n) * 16.0, st,
                (k_restrict_p1<T><<<p1r, kPlaneThreads, 0, st>>>(v.n, B, v.r, w.g, act)));
  else if (red)
    MLMC_LAUNCH(Names<T>::restrict_, rbytes, Ba * interior(w.n) * 26.0, st,
                (k_restrict_red<T><<<fwr, kPlaneThreads, 0, st>>>(v.n, B, v.r, w.g, act)));
  else
    MLMC_LAUNCH(Names<T>::restrict_, rbytes, Ba * interior(w.n) * 54.0, st,
                (k_restrict<T><<<fwr, kPlaneThreads, 0, st>>>(v.n, B, v.r, w.g, act)));
  clear_guess(H, j + 1, nu1, st);
  vcycle(H, j + 1, nu1, nu2, st, true);
  prolong_level(H, j, nu2 > 0, st);
  smooth(nu2, false);
}

// Runs one V-cycle, as a CUDA graph when enabled: the first call captures the cycle's
// launches (counted by the launch tape on every replay), later calls replay it.
inline bool graphs_allowed() {
  static const bool off = [] {
    const char* e = getenv("MLMC_NO_GRAPHS");
    return e && e[0] == '1';
  }();
  return !off;
}

inline bool fmg_graphs() {
  static const bool on = [] {
    const char* e = getenv("MLMC_FMG_GRAPHS");
    return e && e[0] == '1';
  }();
  return on;
}

template <typename T>
struct GraphRunner {
  bool enabled = false;
  cudaGraphExec_t exec = nullptr;
  prof::Tape tape;
  int cap_act = 1;  // active samples when the cycle was captured (its tape's accounting)
  ~GraphRunner() {
    if (exec) cudaGraphExecDestroy(exec);
  }
  // one V-cycle from grid j0, from a zero guess or not, with its first red pass or without (the
  // same on every call of one runner)
  int run(Hier<T>& H, int nu1, int nu2, cudaStream_t st, bool zero, int j0 = 0, bool red_done = false) {
    if (!enabled) {
      vcycle<T>(H, j0, nu1, nu2, st, zero, red_done);
      MLMC_CUDA_TRY(H.failed);
      return MLMC_OK;
    }
    if (!exec) {
      std::shared_lock<std::shared_mutex> lk(capture_lock());
      MLMC_CUDA_TRY(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
      prof::tape_begin();
      vcycle<T>(H, j0, nu1, nu2, st, zero, red_done);
      tape = prof::tape_end();
      cap_act = H.n_act > 0 ? H.n_act : 1;
      cudaGraph_t graph = nullptr;
      MLMC_CUDA_TRY(cudaStreamEndCapture(st, &graph));
      if (H.failed != cudaSuccess) {
        cudaGraphDestroy(graph);
        MLMC_CUDA_TRY(H.failed);
      }
      const cudaError_t e = cudaGraphInstantiate(&exec, graph, 0);
      cudaGraphDestroy(graph);
      if (e != cudaSuccess) {
        exec = nullptr;
        set_error("cudaGraphInstantiate failed: %s", cudaGetErrorString(e));
        return MLMC_ERR_CUDA;
      }
    }
    prof::tape_replay(tape, (double)H.n_act / (double)cap_act);
    MLMC_CUDA_TRY(cudaGraphLaunch(exec, st));
    return MLMC_OK;
  }
};

// The vector kernels of flexible CG on the finest grid, FP64, with the V-cycle's result z read
// where the cycle left it (MIX: FP32, SPLIT: in colour-split storage).
template <typename T, bool SPLIT>
struct CgVectors {
  static constexpr bool MIX = sizeof(T) == 4;
  const Hier<T>& H;
  double* x;
  cudaStream_t st;
  double rtol;
  int maxc;
  int n() const { return H.lv[0].n; }
  const void* z() const { return H.lv[0].u; }
  double all() const { return (double)H.n_act * H.lv[0].n3; }
  dim3 planes() const { return plane_grid(n() * n(), (long long)H.B * n()); }
  void update() const {
    MLMC_LAUNCH("cg_update", all() * 32.0, all() * 6.0, st,
                (k_cg_update<MIX, SPLIT><<<dim3(H.NBu, H.B), kThreads, 0, st>>>(
                    n(), H.alpha, H.Q, H.R, PrecondZ<MIX, SPLIT>{z()}, MIX ? (float*)(void*)H.lv[0].g : nullptr,
                    H.partial, H.part2, H.rzo, H.g2, H.relres, H.cycles, H.active, H.cand, rtol, maxc, H.n_active,
                    H.tick)));
  }
  void dot(bool first) const {
    MLMC_LAUNCH("cg_precond_dot", all() * (MIX ? 12.0 : 16.0), all() * 2.0, st,
                (k_precond_dot<MIX, SPLIT><<<dim3(H.NB, H.B), kThreads, 0, st>>>(
                    n(), PrecondZ<MIX, SPLIT>{z()}, H.R, H.partial, first ? 1 : 0, H.rzo, H.rz, H.beta, H.tick,
                    H.active)));
  }
  void direction(bool first) const {
    MLMC_LAUNCH("cg_p_update", all() * (first ? 12.0 : (MIX ? 36.0 : 40.0)), all() * (first ? 0.0 : 4.0), st,
                (k_p_update<MIX, SPLIT><<<planes(), kPlaneThreads, 0, st>>>(n(), H.B, first ? 1 : 0, H.alpha, H.beta,
                                                                           z(), H.P, x, H.active)));
  }
  void finish(int count) const {
    MLMC_LAUNCH("cg_finish", (double)count * H.lv[0].n3 * 24.0, (double)count * H.lv[0].n3 * 2.0, st,
                (k_cg_finish<<<planes(), kPlaneThreads, 0, st>>>(n(), H.B, H.alpha, H.P, x, H.cand)));
  }
};

// Flexible preconditioned CG: per iteration one operator application with p.q, one residual
// update with r.r and r.z, the V-cycle, one dot product r.z, one update of x and p: 128 bytes and
// 14 FP64 operations per node in mixed precision (an FP64 copy of z, and x updated beside r, made
// it 152), one launch for the scalars (last_block does the others). The FP64 pipe bounds the
// application (1.07 of the 1.06 TFLOP/s the FMA probe reaches at 257^3), HBM p's and x's update
// (5.7 TB/s); r's update, 32 bytes and three FP64 operations per node, is bound by neither alone.
// Per iteration at 257^3: 663 us of vector kernels and three of scalars -> 560. The mixed 257^3
// solve 24.3 -> 22.1 ms, the 257^3 / 129^3 level of two 41.0 -> 39.0.
template <typename T, bool SPLIT>
int pcg_loop(Hier<T>& H, const MGSolveArgs& a, int nu1, int nu2, double rtol, int maxc, cudaStream_t st,
             GraphRunner<T>& gr) {
  const bool mixed = a.cfg.precision == MLMC_PREC_MIXED;
  const int B = H.B, n = a.n;
  Level<T>& l0 = H.lv[0];
  const CgVectors<T, SPLIT> V{H, a.u, st, rtol, maxc};
  const unsigned sb = (B + 3) / 4;  // 128-thread blocks, one warp per sample
  const unsigned g0 = blocks_for((size_t)B * l0.n3, kThreads);
  int azslab = 0;
  const int aslabs = apply_slabs(n, &azslab), NBa = apply_blocks(n);
  const dim3 ag((unsigned)((n * n + 127) / 128), (unsigned)aslabs, (unsigned)B);
  // the outer operator is FP64 in both precisions: the FP64 faces of the finest grid
  const double* D = mixed ? H.D64 : (const double*)(const void*)l0.D;
  const double* Fx = mixed ? H.K64x : (const double*)(const void*)l0.Kx;
  const double* Fy = mixed ? H.K64y : (const double*)(const void*)l0.Ky;
  const double* Fz = mixed ? H.K64z : (const double*)(const void*)l0.Kz;
  auto sync_count = [&](int* out) -> int {
    MLMC_CUDA_TRY(cudaMemcpyAsync(out, H.n_active, sizeof(int), cudaMemcpyDeviceToHost, st));
    MLMC_CUDA_TRY(cudaStreamSynchronize(st));
    return MLMC_OK;
  };
  // z = M r: one V-cycle from zero on the (FP32 copy of the) residual
  auto precondition = [&]() -> int {
    MLMC_CUDA_TRY(clear_guess(H, 0, nu1, st));
    return gr.run(H, nu1, nu2, st, true);
  };
  // r = g - A x, ||r||
  double nodes = H.n_act * interior(n);
  MLMC_CUDA_TRY(cudaMemsetAsync(H.tick, 0, B * sizeof(int), st));
  MLMC_CUDA_TRY(cudaMemsetAsync(H.n_active, 0, sizeof(int), st));
  MLMC_LAUNCH("cg_residual", nodes * (3 * 8.0 + 32), nodes * 16.0, st,
              (k_residual_z<double, double, double, double><<<ag, 128, 0, st>>>(n, azslab, Fx, Fy, Fz, D, H.g64,
                                                                               a.u, H.R, H.partial, H.active)));
  MLMC_LAUNCH("norm_update", B * NBa * 8.0, B * NBa * 1.0, st,
              (k_norm_update<<<sb, 128, 0, st>>>(B, NBa, H.partial, H.g2, H.relres, H.cycles, H.active, 1, 0, rtol,
                                                 maxc, H.n_active)));
  MLMC_TRY(sync_count(&H.n_act));
  if (H.n_act == 0) return MLMC_OK;
  if (mixed && SPLIT)
    MLMC_LAUNCH("to_f32", V.all() * 12.0, 0.0, st,
                (k_to_f32_split<<<V.planes(), kPlaneThreads, 0, st>>>(n, B, H.R, (float*)(void*)l0.g)));
  else if (mixed)
    MLMC_LAUNCH("to_f32", V.all() * 12.0, 0.0, st,
                (k_to_f32<<<g0, kThreads, 0, st>>>((size_t)B * l0.n3, H.R, (float*)(void*)l0.g)));
  MLMC_TRY(precondition());
  V.dot(true);
  V.direction(true);
  while (true) {
    nodes = H.n_act * interior(n);
    MLMC_LAUNCH("cg_apply_dot", nodes * 48.0, nodes * 16.0, st,
                (k_apply_dot_z<double, double><<<ag, 128, 0, st>>>(n, azslab, Fx, Fy, Fz, D, H.P, H.Q, H.part_apply,
                                                                    H.active)));
    MLMC_LAUNCH("cg_scalar", B * NBa * 8.0, 0.0, st,
                (k_cg_alpha<<<sb, 128, 0, st>>>(B, NBa, H.part_apply, H.rz, H.alpha, H.active)));
    MLMC_CUDA_TRY(cudaMemsetAsync(H.n_active, 0, sizeof(int), st));
    V.update();
    int na = 0;
    MLMC_TRY(sync_count(&na));
    const int done = H.n_act - na;
    H.n_act = na;
    if (done > 0) V.finish(done);
    if (na == 0) break;
    MLMC_TRY(precondition());
    V.dot(false);
    V.direction(false);
  }
  return MLMC_OK;
}

// ---------------------------------------------------------------------------------
// Small-grid engine (MLMC_ENGINE_CTA): one persistent launch runs the whole solve of a
// batch on grids up to 33^3. Each CTA takes the next sample from a device counter and
// runs that sample's cycles to convergence -- V-cycles, convergence tests, and the CG
// recurrences -- with block barriers between the phases instead of kernel launches and
// without host round trips. Every node update uses the operations of the batched
// kernels in their order, and every per-sample sum uses the batched kernels' partition
// (column z-march blocks of 128 threads, flat chunks of 256 threads) and reduction trees,
// so a sample's iterates, cycle count and residuals are bit for bit those of the batched
// path.
// ---------------------------------------------------------------------------------
constexpr int kCtaThreads = 256;

// MLMC_ENGINE_CTA where it applies (finite volumes, stationary cycles, refinement or CG,
// grids up to 33^3); MLMC_ENGINE_AUTO takes it for grids up to 17^3 (measured 1.15-1.4x
// faster than the batched engine at every batch size from 1 to 4096 samples, with 16-20x
// fewer launches); a 33^3 sample is too much work for one CTA (0.45-0.97x).
inline bool cta_engine_chosen(const mg_cfg& c, int n, int B) {
  const bool ok = c.disc == MLMC_DISC_FV && c.accel != MLMC_ACCEL_FMG && n <= kCtaMaxN;
  if (!ok || c.engine == MLMC_ENGINE_BATCHED) return false;
  if (c.engine == MLMC_ENGINE_CTA) return true;
  static const int env = [] {
    const char* e = getenv("MLMC_ENGINE");
    return e ? atoi(e) : 0;
  }();
  if (env == MLMC_ENGINE_BATCHED) return false;
  if (env == MLMC_ENGINE_CTA) return true;
  // measured: 17^3 1.15-1.4x the batched kernels at 1..4096 samples; 33^3 about even at
  // 1024 samples (FP64 stationary: 73.6 against 74.8 ms, 34 against 757 launches) and
  // slower below (256 samples of mixed CG: 31.0 against 24.8 ms; one CTA per sample leaves
  // SMs idle while fewer samples than resident CTAs remain)
  return n <= 17 || (n <= 33 && B >= 1024);
}
constexpr int kCtaMaxPartials = 64;

template <typename T>
struct CtaLevel {
  int n = 0;
  const T *Kx = nullptr, *Ky = nullptr, *Kz = nullptr, *D = nullptr, *Dinv = nullptr;
  const T* kn = nullptr;  // reciprocal nodal coefficient (FP32 nodal sweep), else nullptr
  T *u = nullptr, *g = nullptr, *r = nullptr;
};

enum { kCtaStationary = 0, kCtaRefinement = 1, kCtaCG = 2 };

template <typename T>
struct CtaArgs {
  int L = 0, B = 0, nu1 = 2, nu2 = 2, maxc = 1, mode = 0;
  double rtol = 0.0, red_limit = 0.0;
  int red_fused = 0;
  CtaLevel<T> lv[4];
  const double* Ainv = nullptr;
  // outer FP64 operator (FP64 faces and diagonal of the finest grid), right-hand side, iterate
  const double *Fx = nullptr, *Fy = nullptr, *Fz = nullptr, *D = nullptr, *g64 = nullptr;
  double* x = nullptr;
  double *R = nullptr, *P = nullptr, *Q = nullptr, *Z = nullptr;  // CG vectors (Z: mixed only)
  const double* g2 = nullptr;
  double* relres = nullptr;
  int *cycles = nullptr, *active = nullptr, *work = nullptr;
  int NB = 1, zslab = 1, slabs = 1;  // flat-chunk partials per sample; column z-march geometry
};

// block_sum<128> of one half of a 256-thread CTA (threads 128 h .. 128 h + 127): the same
// shuffle tree; valid in thread 128 h. Both halves must call it together.
__device__ __forceinline__ double half_block_sum128(double v, double* warp_part8) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, h = threadIdx.x >> 7;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) warp_part8[wid] = v;
  __syncthreads();
  double r = 0.0;
  if ((wid & 3) == 0) {
    r = lane < 4 ? warp_part8[4 * h + lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  return r;
}

template <typename T, bool ZERO = false>
__device__ void cta_smooth(const CtaLevel<T>& v, int s, int colour) {
  const int n = v.n, m = n - 2, half = (n - 1) / 2, lh = 31 - __clz(half), per = m * half;
  const size_t n3 = (size_t)n * n * n, n2 = (size_t)n * n;
  for (int it = threadIdx.x; it < per * m; it += blockDim.x) {
    const int zi = it / per, q = it - zi * per;
    const int xi = q & (half - 1), y = 1 + (q >> lh), z = 1 + zi;
    const int x = (((1 + y + z) & 1) == colour ? 1 : 2) + 2 * xi;
    if (x > n - 2) continue;
    const size_t p = (size_t)s * n3 + (size_t)(z * n * n + y * n + x);
    if constexpr (sizeof(T) == 4) {
      if (v.kn) {
        const float* kn = (const float*)v.kn;
        float* u = (float*)v.u;
        const float kc = kn[p];
        const float kxm = nodal_face(kn[p - 1], kc), kxp = nodal_face(kc, kn[p + 1]);
        const float kym = nodal_face(kn[p - n], kc), kyp = nodal_face(kc, kn[p + n]);
        const float kzm = nodal_face(kn[p - n2], kc), kzp = nodal_face(kc, kn[p + n2]);
        float d = kxm;
        d += kxp;
        d += kym;
        d += kyp;
        d += kzm;
        d += kzp;
        const float dinv = __fdividef(1.0f, d);
        float acc = ((const float*)v.g)[p];
        if (!ZERO) {
          acc = fmaf(kxm, u[p - 1], acc);
          acc = fmaf(kxp, u[p + 1], acc);
          acc = fmaf(kym, u[p - n], acc);
          acc = fmaf(kyp, u[p + n], acc);
          acc = fmaf(kzm, u[p - n2], acc);
          acc = fmaf(kzp, u[p + n2], acc);
        }
        u[p] = acc * dinv;
        continue;
      }
    }
    T* u = v.u;
    T acc = v.g[p];
    if (!ZERO) {
      acc = fma(v.Kx[p - 1], u[p - 1], acc);
      acc = fma(v.Kx[p], u[p + 1], acc);
      acc = fma(v.Ky[p - n], u[p - n], acc);
      acc = fma(v.Ky[p], u[p + n], acc);
      acc = fma(v.Kz[p - n2], u[p - n2], acc);
      acc = fma(v.Kz[p], u[p + n2], acc);
    }
    u[p] = acc * v.Dinv[p];
  }
}

// in-cycle residual r~ (k_residual_z / k_residual_nodal operations), 0 on the boundary; RED:
// at the red nodes only (k_residual_red)
template <typename T, bool RED>
__device__ void cta_residual(const CtaLevel<T>& v, int s) {
  const int n = v.n, half = (n + 1) / 2, row = RED ? half : n;
  const size_t n3 = (size_t)n * n * n, n2 = (size_t)n * n;
  for (int i = threadIdx.x; i < row * n * n; i += blockDim.x) {
    const int z = i / (row * n), rem = i - z * row * n, y = rem / row, xq = rem - y * row;
    const int x = RED ? 2 * xq + ((y + z) & 1) : xq;
    if (RED && x > n - 1) continue;
    const size_t p = (size_t)s * n3 + (size_t)((z * n + y) * n + x);
    T rr = T(0);
    if (x > 0 && y > 0 && z > 0 && x < n - 1 && y < n - 1 && z < n - 1) {
      bool done = false;
      if constexpr (sizeof(T) == 4) {
        if (v.kn) {
          const float* kn = (const float*)v.kn;
          const float* u = (const float*)v.u;
          const float kc = kn[p];
          const float kxm = nodal_face(kn[p - 1], kc), kxp = nodal_face(kc, kn[p + 1]);
          const float kym = nodal_face(kn[p - n], kc), kyp = nodal_face(kc, kn[p + n]);
          const float kzm = nodal_face(kn[p - n2], kc), kzp = nodal_face(kc, kn[p + n2]);
          float d = kxm;
          d += kxp;
          d += kym;
          d += kyp;
          d += kzm;
          d += kzp;
          float q = fmaf(-d, u[p], ((const float*)v.g)[p]);
          q = fmaf(kxm, u[p - 1], q);
          q = fmaf(kxp, u[p + 1], q);
          q = fmaf(kym, u[p - n], q);
          q = fmaf(kyp, u[p + n], q);
          q = fmaf(kzm, u[p - n2], q);
          q = fmaf(kzp, u[p + n2], q);
          rr = (T)q;
          done = true;
        }
      }
      if (!done) {
        const T* u = v.u;
        rr = fma(-v.D[p], u[p], v.g[p]);
        rr = fma(v.Kx[p - 1], u[p - 1], rr);
        rr = fma(v.Kx[p], u[p + 1], rr);
        rr = fma(v.Ky[p - n], u[p - n], rr);
        rr = fma(v.Ky[p], u[p + n], rr);
        rr = fma(v.Kz[p - n2], u[p - n2], rr);
        rr = fma(v.Kz[p], u[p + n2], rr);
      }
    }
    v.r[p] = rr;
  }
}

// g_c = 4 FW(r~) at interior coarse nodes (k_restrict's operations; RED: k_restrict_red's) and
// u_c = 0 where the coarse grid's first pass reads it (without pre-smoothing: !RED)
template <typename T, bool RED>
__device__ void cta_restrict(const CtaLevel<T>& v, const CtaLevel<T>& w, int s) {
  const int nf = v.n, nc = w.n, mc = nc - 2;
  const size_t nf3 = (size_t)nf * nf * nf, nc3 = (size_t)nc * nc * nc;
  const int nf2 = nf * nf;
  if (!RED)
    for (int i = threadIdx.x; i < (int)nc3; i += blockDim.x) w.u[(size_t)s * nc3 + i] = T(0);
  for (int i = threadIdx.x; i < mc * mc * mc; i += blockDim.x) {
    const int Z = 1 + i / (mc * mc), rem = i - (Z - 1) * mc * mc, Y = 1 + rem / mc, X = 1 + rem - (Y - 1) * mc;
    const T* rb = v.r + (size_t)s * nf3 + (size_t)(2 * Z * nf2 + 2 * Y * nf + 2 * X);
    T acc = 0;
#pragma unroll
    for (int dz = -1; dz <= 1; ++dz)
#pragma unroll
      for (int dy = -1; dy <= 1; ++dy)
#pragma unroll
        for (int dx = -1; dx <= 1; ++dx) {
          if (RED && ((dx + dy + dz) & 1)) continue;
          const T wgt = (T)((2 - abs(dx)) * (2 - abs(dy)) * (2 - abs(dz))) * (T)(1.0 / 16.0);
          acc = fma(wgt, rb[dz * nf2 + dy * nf + dx], acc);
        }
    w.g[(size_t)s * nc3 + (size_t)((Z * nc + Y) * nc + X)] = acc;
  }
}

// u_f += trilinear interpolation of e_c (k_prolong's operations; BLACK: at the black nodes)
template <typename T, bool BLACK>
__device__ void cta_prolong(const CtaLevel<T>& w, const CtaLevel<T>& v, int s) {
  // one coarse cell per thread (k_prolong_blk's sums, bit for bit k_prolong's)
  const int nf = v.n, nc = w.n, mc = nc - 1;
  const size_t nf3 = (size_t)nf * nf * nf, nc3 = (size_t)nc * nc * nc, nc2 = (size_t)nc * nc;
  for (int i = threadIdx.x; i < mc * mc * mc; i += blockDim.x) {
    const int Z = i / (mc * mc), rem = i - Z * mc * mc, Y = rem / mc, X = rem - Y * mc;
    const T* e = w.u + (size_t)s * nc3 + (size_t)((Z * nc + Y) * nc + X);
    const T c[8] = {e[0], e[1], e[nc], e[nc + 1], e[nc2], e[nc2 + 1], e[nc2 + nc], e[nc2 + nc + 1]};
    T val[8];
    prolong_block_sums(c, val);
    T* ub = v.u + (size_t)s * nf3;
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int dx = k & 1, dy = (k >> 1) & 1, dz = k >> 2;
      if (BLACK && !((dx + dy + dz) & 1)) continue;
      const int x = 2 * X + dx, y = 2 * Y + dy, z = 2 * Z + dz;
      if (x < 1 || y < 1 || z < 1 || x > nf - 2 || y > nf - 2 || z > nf - 2) continue;
      const T wgt = dx + dy + dz == 0 ? T(1) : dx + dy + dz == 1 ? T(0.5) : dx + dy + dz == 2 ? T(0.25) : T(0.125);
      ub[(size_t)((z * nf + y) * nf + x)] += wgt * val[k];
    }
  }
}

// zero: the finest iterate is zero on entry (its interior need not be: with pre-smoothing
// the first red pass does not read it)
// red_done: the finest grid's first red pass has been taken (cta_red_pass_norm)
template <typename T>
__device__ void cta_vcycle(const CtaArgs<T>& A, int s, bool zero, bool red_done = false) {
  // down: smoothing, residual, restriction
  for (int j = 0; j < A.L - 1; ++j) {
    for (int k = 0; k < A.nu1; ++k)
      for (int c = 0; c < 2; ++c) {
        if (red_done && j == 0 && k == 0 && c == 0) continue;
        if (k == 0 && c == 0 && (j > 0 || zero))
          cta_smooth<T, true>(A.lv[j], s, c);
        else
          cta_smooth<T, false>(A.lv[j], s, c);
        __syncthreads();
      }
    if (A.nu1 > 0)
      cta_residual<T, true>(A.lv[j], s);
    else
      cta_residual<T, false>(A.lv[j], s);
    __syncthreads();
    if (A.nu1 > 0)
      cta_restrict<T, true>(A.lv[j], A.lv[j + 1], s);
    else
      cta_restrict<T, false>(A.lv[j], A.lv[j + 1], s);
    __syncthreads();
  }
  // exact solve on the 5^3 grid (k_coarse_apply)
  {
    const CtaLevel<T>& v = A.lv[A.L - 1];
    const int i = threadIdx.x;
    if (i < 27) {
      const double* X = A.Ainv + (size_t)s * 729 + (size_t)i * 27;
      const size_t base = (size_t)s * 125;
      double val = 0.0;
      for (int q = 0; q < 27; ++q) {
        const int x = 1 + q % 3, y = 1 + (q / 3) % 3, z = 1 + q / 9;
        val = fma(X[q], (double)v.g[base + (z * 5 + y) * 5 + x], val);
      }
      const int x = 1 + i % 3, y = 1 + (i / 3) % 3, z = 1 + i / 9;
      v.u[base + (z * 5 + y) * 5 + x] = (T)val;
    }
    __syncthreads();
  }
  // up: correction, smoothing
  for (int j = A.L - 2; j >= 0; --j) {
    if (A.nu2 > 0)
      cta_prolong<T, true>(A.lv[j + 1], A.lv[j], s);
    else
      cta_prolong<T, false>(A.lv[j + 1], A.lv[j], s);
    __syncthreads();
    for (int k = 0; k < A.nu2; ++k)
      for (int c = 0; c < 2; ++c) {
        cta_smooth<T, false>(A.lv[j], s, c);
        __syncthreads();
      }
  }
}

// Column z-march partials (k_residual_z / k_apply_dot_z partition, 128-thread blocks, two
// per pass of the CTA): APPLY = false: r~ = g - D x + sum K x_q (stored as TR into r when
// r != nullptr) and partials of r~^2; APPLY = true: q = D p - sum K p_q and partials of
// p.q. Returns the total of the partials (k_norm_update / k_cg_scalar's warp tree).
template <bool APPLY, typename TR>
__device__ double cta_zmarch(const double* __restrict__ Fx, const double* __restrict__ Fy,
                             const double* __restrict__ Fz, const double* __restrict__ D,
                             const double* __restrict__ g, const double* __restrict__ x, TR* __restrict__ r, int n,
                             int zslab, int slabs, int s, double* part, double* warp_part8, double* bcast) {
  const int CB = (n * n + 127) / 128, nb = CB * slabs, h = threadIdx.x >> 7, t = threadIdx.x & 127;
  const size_t n2 = (size_t)n * n;
  for (int vb0 = 0; vb0 < nb; vb0 += 2) {
    const int vb = vb0 + h;
    double acc = 0.0;
    if (vb < nb) {
      const int cb = vb % CB, slab = vb / CB;
      const int c = cb * 128 + t;
      const int zlo = 1 + slab * zslab, zhi = min(n - 2, zlo + zslab - 1);
      if (c < n * n) {
        const int y = c / n, xx = c - y * n;
        const size_t col = (size_t)s * n2 * n + c;
        if (xx > 0 && y > 0 && xx < n - 1 && y < n - 1) {
          double pm = x[col + (size_t)(zlo - 1) * n2], pc = x[col + (size_t)zlo * n2];
          double kzm = Fz[col + (size_t)(zlo - 1) * n2];
          for (int z = zlo; z <= zhi; ++z) {
            const size_t p = col + (size_t)z * n2;
            const double pp = x[p + n2];
            const double kzp = Fz[p];
            if (APPLY) {
              double v = D[p] * pc;
              v = fma(-Fx[p - 1], x[p - 1], v);
              v = fma(-Fx[p], x[p + 1], v);
              v = fma(-Fy[p - n], x[p - n], v);
              v = fma(-Fy[p], x[p + n], v);
              v = fma(-kzm, pm, v);
              v = fma(-kzp, pp, v);
              acc = fma(pc, v, acc);
              r[p] = (TR)v;
            } else {
              double rr = fma(-D[p], pc, g[p]);
              rr = fma(Fx[p - 1], x[p - 1], rr);
              rr = fma(Fx[p], x[p + 1], rr);
              rr = fma(Fy[p - n], x[p - n], rr);
              rr = fma(Fy[p], x[p + n], rr);
              rr = fma(kzm, pm, rr);
              rr = fma(kzp, pp, rr);
              if (r) r[p] = (TR)rr;
              acc += rr * rr;
            }
            pm = pc;
            pc = pp;
            kzm = kzp;
          }
        } else if (r) {
          for (int z = zlo; z <= zhi; ++z) r[col + (size_t)z * n2] = TR(0);
        }
        if (r && slab == 0) r[col] = TR(0);
        if (r && slab == slabs - 1) r[col + (size_t)(n - 1) * n2] = TR(0);
      }
    }
    const double bs = half_block_sum128(acc, warp_part8);
    if (t == 0 && vb < nb) part[vb] = bs;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const double tot = warp_sum_partials(part, nb);
    if (threadIdx.x == 0) *bcast = tot;
  }
  __syncthreads();
  return *bcast;
}

// The finest grid's red pass of sample s (cta_smooth's operations) with the sum of the squared red
// residuals it passes by (k_rbgs_norm_split), the same in every thread; the replaced values go to
// the grid's residual array, which the cycle has not written yet.
template <typename T>
__device__ double cta_red_pass_norm(const CtaLevel<T>& v, int s, double* bcast) {
  const int n = v.n, m = n - 2, half = (n - 1) / 2, lh = 31 - __clz(half), per = m * half;
  const size_t n3 = (size_t)n * n * n, n2 = (size_t)n * n;
  T* u = v.u;
  double sq = 0.0;
  for (int it = threadIdx.x; it < per * m; it += kCtaThreads) {
    const int zi = it / per, q = it - zi * per;
    const int xi = q & (half - 1), y = 1 + (q >> lh), z = 1 + zi;
    const int xx = 1 + ((y + z + 1) & 1) + 2 * xi;
    if (xx > n - 2) continue;
    const size_t p = (size_t)s * n3 + (size_t)(z * n * n + y * n + xx);
    T acc = v.g[p];
    acc = fma(v.Kx[p - 1], u[p - 1], acc);
    acc = fma(v.Kx[p], u[p + 1], acc);
    acc = fma(v.Ky[p - n], u[p - n], acc);
    acc = fma(v.Ky[p], u[p + n], acc);
    acc = fma(v.Kz[p - n2], u[p - n2], acc);
    acc = fma(v.Kz[p], u[p + n2], acc);
    const T up = u[p], rr = fma(-v.D[p], up, acc);
    sq += (double)rr * (double)rr;
    v.r[p] = up;
    u[p] = acc * v.Dinv[p];
  }
  const double b = block_sum<kCtaThreads>(sq);
  __syncthreads();
  if (threadIdx.x == 0) *bcast = b;
  __syncthreads();
  return *bcast;
}

// Puts the replaced red values back.
template <typename T>
__device__ void cta_restore_red(const CtaLevel<T>& v, int s) {
  const int n = v.n, m = n - 2;
  const size_t b = (size_t)s * n * n * n;
  for (int it = threadIdx.x; it < m * m * m; it += kCtaThreads) {
    const int z = 1 + it / (m * m), q = it - (z - 1) * m * m, y = 1 + q / m, x = 1 + q - (y - 1) * m;
    const size_t p = b + (size_t)((z * n + y) * n + x);
    if (!((x + y + z) & 1)) v.u[p] = v.r[p];
  }
  __syncthreads();
}

// convergence bookkeeping of one sample (k_norm_update, mode 1); returns the active flag
__device__ __forceinline__ int cta_norm_update(double t, double g2, double rtol, int maxc, int inc, double* rel,
                                               int* cyc) {
  *rel = g2 > 0.0 ? sqrt(t / g2) : 0.0;
  *cyc += inc;
  return (rtol > 0.0) ? (*rel > rtol && *cyc < maxc) : (*cyc < maxc);
}

template <typename T>
__global__ void __launch_bounds__(kCtaThreads) k_solve_cta(CtaArgs<T> A) {
  __shared__ double part[kCtaMaxPartials], part2[kCtaMaxPartials], warp_part8[8], bcast[1];
  __shared__ int s_next;
  const int n = A.lv[0].n;
  const size_t n3 = (size_t)n * n * n;
  const unsigned chunk = ((unsigned)n3 + A.NB - 1) / A.NB;
  for (;;) {
    if (threadIdx.x == 0) s_next = atomicAdd(A.work, 1);
    __syncthreads();
    const int s = s_next;
    __syncthreads();
    if (s >= A.B) return;
    const double g2 = A.g2[s];
    double rel = 0.0;
    int cyc = 0, act = 0;
    if (A.mode == kCtaStationary) {
      // FP64 V-cycles on the level-0 iterate until the residual test passes
      for (int inc = 0;; inc = 1) {
        // after a cycle the red residuals, taken along with the next cycle's first red pass, decide
        // whether the sample goes on; the full one whether it is done (the batched test); fixed
        // cycles need the last residual alone
        bool go = inc > 0 && A.rtol <= 0.0 && cyc + 1 < A.maxc, red_done = false;
        if (inc > 0 && A.red_fused && A.nu1 > 0 && A.L > 1 && cyc + 1 < A.maxc) {
          const double tr = cta_red_pass_norm<T>(A.lv[0], s, bcast);
          go = red_done = g2 > 0.0 && sqrt(tr / g2) > A.red_limit;
          if (!go) cta_restore_red<T>(A.lv[0], s);
        }
        if (go) {
          ++cyc;
        } else {
          const double t = cta_zmarch<false, double>(A.Fx, A.Fy, A.Fz, A.D, A.g64, A.x, (double*)nullptr, n, A.zslab,
                                                     A.slabs, s, part, warp_part8, bcast);
          act = cta_norm_update(t, g2, A.rtol, A.maxc, inc, &rel, &cyc);
          if (!act) break;
        }
        cta_vcycle(A, s, false, red_done);
      }
    } else if (A.mode == kCtaRefinement) {
      // FP32 V-cycles on FP64 residuals: r32 = g - A x, e = V(r32), x += e
      CtaLevel<T>& l0 = A.lv[0];
      for (int inc = 0;; inc = 1) {
        const double t = cta_zmarch<false, T>(A.Fx, A.Fy, A.Fz, A.D, A.g64, A.x, l0.g, n, A.zslab, A.slabs, s, part,
                                              warp_part8, bcast);
        act = cta_norm_update(t, g2, A.rtol, A.maxc, inc, &rel, &cyc);
        if (!act) break;
        if (A.nu1 == 0) {
          for (size_t i = threadIdx.x; i < n3; i += blockDim.x) l0.u[(size_t)s * n3 + i] = T(0);
          __syncthreads();
        }
        cta_vcycle(A, s, true);
        for (size_t i = threadIdx.x; i < n3; i += blockDim.x) A.x[(size_t)s * n3 + i] += widen(l0.u[(size_t)s * n3 + i]);
        __syncthreads();
      }
    } else {
      // flexible preconditioned CG (pcg_loop's recurrences)
      CtaLevel<T>& l0 = A.lv[0];
      const bool mixed = sizeof(T) == 4;
      double* zv = mixed ? A.Z : (double*)(void*)l0.u;
      const size_t b0 = (size_t)s * n3;
      double rz = 0.0, rzo = 0.0, alpha = 0.0, beta = 0.0;
      // z = M r and the partials of r.z (flat chunks): the preconditioner
      auto precondition = [&]() -> double {
        if (A.nu1 == 0) {
          for (size_t i = threadIdx.x; i < n3; i += blockDim.x) l0.u[b0 + i] = T(0);
          __syncthreads();
        }
        cta_vcycle(A, s, true);
        for (int b = 0; b < A.NB; ++b) {
          const unsigned lo = b * chunk, hi = lo + chunk < (unsigned)n3 ? lo + chunk : (unsigned)n3;
          double acc = 0.0;
          for (unsigned i = lo + threadIdx.x; i < hi; i += kCtaThreads) {
            const size_t t = b0 + i;
            double z;
            if (mixed) {
              z = widen(((const float*)(const void*)l0.u)[t]);
              zv[t] = z;
            } else {
              z = zv[t];
            }
            acc = fma(A.R[t], z, acc);
          }
          const double bsum = block_sum<kCtaThreads>(acc);
          if (threadIdx.x == 0) part[b] = bsum;
        }
        __syncthreads();
        if (threadIdx.x < 32) {
          const double tot = warp_sum_partials(part, A.NB);
          if (threadIdx.x == 0) *bcast = tot;
        }
        __syncthreads();
        return *bcast;
      };
      const double t0 = cta_zmarch<false, double>(A.Fx, A.Fy, A.Fz, A.D, A.g64, A.x, A.R, n, A.zslab, A.slabs, s,
                                                  part, warp_part8, bcast);
      act = cta_norm_update(t0, g2, A.rtol, A.maxc, 0, &rel, &cyc);
      if (act) {
        if (mixed)
          for (size_t i = threadIdx.x; i < n3; i += blockDim.x) ((float*)(void*)l0.g)[b0 + i] = (float)A.R[b0 + i];
        __syncthreads();
        rz = precondition();
        for (size_t i = threadIdx.x; i < n3; i += blockDim.x) A.P[b0 + i] = zv[b0 + i];
        __syncthreads();
        for (;;) {
          const double pq = cta_zmarch<true, double>(A.Fx, A.Fy, A.Fz, A.D, nullptr, A.P, A.Q, n, A.zslab, A.slabs, s,
                                                     part, warp_part8, bcast);
          alpha = pq != 0.0 ? rz / pq : 0.0;
          // x += alpha p, r -= alpha q; partials of r.r and r.z_old (flat chunks)
          for (int b = 0; b < A.NB; ++b) {
            const unsigned lo = b * chunk, hi = lo + chunk < (unsigned)n3 ? lo + chunk : (unsigned)n3;
            double rr = 0.0, rzp = 0.0;
            for (unsigned i = lo + threadIdx.x; i < hi; i += kCtaThreads) {
              const size_t t = b0 + i;
              A.x[t] = fma(alpha, A.P[t], A.x[t]);
              const double rn = fma(-alpha, A.Q[t], A.R[t]);
              A.R[t] = rn;
              if (mixed) ((float*)(void*)l0.g)[t] = (float)rn;
              rr = fma(rn, rn, rr);
              rzp = fma(rn, zv[t], rzp);
            }
            const double b1 = block_sum<kCtaThreads>(rr);
            if (threadIdx.x == 0) part[b] = b1;
            const double b2 = block_sum<kCtaThreads>(rzp);
            if (threadIdx.x == 0) part2[b] = b2;
          }
          __syncthreads();
          if (threadIdx.x < 32) {
            const double a1 = warp_sum_partials(part2, A.NB);
            const double a2 = warp_sum_partials(part, A.NB);
            if (threadIdx.x == 0) {
              bcast[0] = a1;
              warp_part8[0] = a2;
            }
          }
          __syncthreads();
          rzo = bcast[0];
          const double trr = warp_part8[0];
          __syncthreads();
          act = cta_norm_update(trr, g2, A.rtol, A.maxc, 1, &rel, &cyc);
          if (!act) break;
          const double rzn = precondition();
          beta = rz != 0.0 ? (rzn - rzo) / rz : 0.0;
          rz = rzn;
          for (size_t i = threadIdx.x; i < n3; i += blockDim.x) A.P[b0 + i] = fma(beta, A.P[b0 + i], zv[b0 + i]);
          __syncthreads();
        }
      }
    }
    if (threadIdx.x == 0) {
      A.relres[s] = rel;
      A.cycles[s] = cyc;
      A.active[s] = act;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------
// The small-grid engine on 17^3 grids: one block of 512 threads per SM with the whole cycle in
// registers and shared memory. A thread owns up to four nodes of either colour for the whole
// solve and keeps their six faces in registers; 1/D, iterate, right-hand side and red residuals of
// 17^3, 9^3 and 5^3 and the 9^3 coefficients are in shared memory (183 KB in FP64, 92 KB in FP32).
// Operations, partitions and trees are k_solve_cta's (which keeps everything in global memory,
// read through L2 in every pass, and serves 9^3 and 33^3), so results are bit for bit the same.
// Bound by the chain of passes, one sample per SM. A served request (one mixed CG sample) takes
// 0.55 ms in this kernel (k_solve_cta 1.12), 0.86 in all. Stored faces only: a form that also took
// 1/k for the nodal sweep through TailGrid's passes gave wrong iterates as ptxas compiles it by
// default, right ones with -Xptxas -O1 or with those passes out of line.
// ---------------------------------------------------------------------------------
template <typename T>
struct Solve17 {
  static constexpr int N = 17;
  using G0 = TailGrid<T, 17, false>;
  using G1 = TailGrid<T, 9, false>;
  static constexpr int items = G0::M * G0::M * G0::HALF, per = (items + kTailThreads - 1) / kTailThreads;
  // shared memory in elements of T: u, g, r of both grids, u and g of 5^3, five 9^3 coefficients,
  // and 1/D of 17^3
  static constexpr size_t elems = (size_t)G0::shared_iter + G1::shared_iter + 250 + 5 * G1::N3 + G0::N3;
  G0 a;
  G1 b;
  T *u5, *g5;
  T c[2][per][6];  // faces -x, +x, -y, +y, -z, +z of the thread's nodes
  const T* D;      // diagonal of the sample (global)

  __device__ __forceinline__ int item(int k, int colour, bool& on) const {  // linear index of node k
    int x, y, z;
    const int it = threadIdx.x + k * kTailThreads;
    on = it < items && G0::node(it, colour, x, y, z);
    return on ? (z * N + y) * N + x : 0;
  }
  __device__ void load(const CtaArgs<T>& A, int s, T* sm) {
    T* p = sm;
    a.u = p;
    a.g = p + G0::N3;
    a.r = p + 2 * G0::N3;
    p += G0::shared_iter;
    b.u = p;
    b.g = p + G1::N3;
    b.r = p + 2 * G1::N3;
    p += G1::shared_iter;
    u5 = p;
    g5 = p + 125;
    p += 250;
    T* const c9 = p;
    p += 5 * G1::N3;
    T* const dinv = p;
    for (int i = threadIdx.x; i < (int)(c9 - sm); i += kTailThreads) sm[i] = T(0);
    const CtaLevel<T>&v = A.lv[0], &w = A.lv[1];
    const size_t o = (size_t)s * G0::N3, o9 = (size_t)s * G1::N3;
    D = v.D + o;
#pragma unroll
    for (int col = 0; col < 2; ++col)
#pragma unroll
      for (int k = 0; k < per; ++k) {
        bool on;
        const size_t q = o + item(k, col, on);
        if (!on) continue;
        c[col][k][0] = v.Kx[q - 1];
        c[col][k][1] = v.Kx[q];
        c[col][k][2] = v.Ky[q - N];
        c[col][k][3] = v.Ky[q];
        c[col][k][4] = v.Kz[q - G0::N2];
        c[col][k][5] = v.Kz[q];
      }
    for (int i = threadIdx.x; i < G0::N3; i += kTailThreads) dinv[i] = v.Dinv[o + i];
    a.Dinv = dinv;
    const T* src[5] = {w.Kx, w.Ky, w.Kz, w.D, w.Dinv};
#pragma unroll
    for (int q = 0; q < 5; ++q)
      for (int i = threadIdx.x; i < G1::N3; i += kTailThreads) c9[q * G1::N3 + i] = src[q][o9 + i];
    a.kn = b.kn = nullptr;
    b.Kx = c9;
    b.Ky = c9 + G1::N3;
    b.Kz = c9 + 2 * G1::N3;
    b.D = c9 + 3 * G1::N3;
    b.Dinv = c9 + 4 * G1::N3;
    __syncthreads();
  }
  __device__ __forceinline__ T faces(const T (&f)[6], int p, T acc) const {
    const T* u = a.u;
    acc = fma(f[0], u[p - 1], acc);
    acc = fma(f[1], u[p + 1], acc);
    acc = fma(f[2], u[p - N], acc);
    acc = fma(f[3], u[p + N], acc);
    acc = fma(f[4], u[p - G0::N2], acc);
    return fma(f[5], u[p + G0::N2], acc);
  }
  template <int COL>
  __device__ void pass(bool zero) {
#pragma unroll
    for (int k = 0; k < per; ++k) {
      bool on;
      const int p = item(k, COL, on);
      if (on) a.u[p] = (zero ? a.g[p] : faces(c[COL][k], p, a.g[p])) * a.Dinv[p];
    }
    __syncthreads();
  }
  // red residuals into r; returns the thread's sum of their squares
  __device__ double red_residual(bool store) {
    double sq = 0.0;
#pragma unroll
    for (int k = 0; k < per; ++k) {
      bool on;
      const int p = item(k, 0, on);
      if (!on) continue;
      const T rr = faces(c[0][k], p, fma(-D[p], a.u[p], a.g[p]));
      if (store) a.r[p >> 1] = rr;
      else sq += (double)rr * (double)rr;
    }
    if (store) __syncthreads();
    return sq;
  }
  // one cycle on a.u for the right-hand side a.g (without pre- or post-smoothing the full
  // residual or interpolation would be needed: k_solve_cta takes those)
  __device__ void cycle(const CtaArgs<T>& A, int s, bool zero) {
    for (int k = 0; k < A.nu1; ++k) {
      pass<0>(zero && k == 0);
      pass<1>(false);
    }
    red_residual(true);
    a.template restrict_to<false>(b.g);
    for (int k = 0; k < A.nu1; ++k) {
      b.pass(0, k == 0);
      b.pass(1, false);
    }
    b.red_residual();
    b.template restrict_to<false>(g5);
    if (threadIdx.x < 27) {  // the exact solve (k_coarse_apply)
      const int i = threadIdx.x;
      const double* X = A.Ainv + (size_t)s * 729 + (size_t)i * 27;
      double v = 0.0;
      for (int q = 0; q < 27; ++q) v = fma(X[q], (double)g5[((1 + q / 9) * 5 + 1 + (q / 3) % 3) * 5 + 1 + q % 3], v);
      u5[((1 + i / 9) * 5 + 1 + (i / 3) % 3) * 5 + 1 + i % 3] = (T)v;
    }
    __syncthreads();
    b.template prolong_from<false>(u5);
    for (int k = 0; k < A.nu2; ++k) {
      b.pass(0, false);
      b.pass(1, false);
    }
    a.template prolong_from<false>(b.u);
    for (int k = 0; k < A.nu2; ++k) {
      pass<0>(false);
      pass<1>(false);
    }
  }
};

// block_sum of each group of 32 W threads: the same trees; valid in the group's first thread.
template <int W>
__device__ __forceinline__ double group_sum(double v, double* warp_part) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if (lane == 0) warp_part[wid] = v;
  __syncthreads();
  double r = 0.0;
  if (wid % W == 0) {
    r = lane < W ? warp_part[wid + lane] : 0.0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  return r;
}

template <typename T>
__global__ void __launch_bounds__(kTailThreads, 1) k_solve17(CtaArgs<T> A) {
  constexpr bool MIX = sizeof(T) == 4;
  constexpr int N = 17, N2 = N * N, N3 = N * N2;
  constexpr int VB = (N2 + 127) / 128;               // k_residual_z's blocks: one z-slab (apply_slabs(17))
  static_assert(VB * 128 <= kTailThreads, "one column per thread");
  extern __shared__ __align__(16) unsigned char tail_smem[];
  __shared__ double part[kCtaMaxPartials], part2[kCtaMaxPartials], warp_part[kTailThreads / 32], bcast[2];
  __shared__ int s_next, cyc, act, go_on;
  __shared__ double rel;
  const int tid = threadIdx.x;
  Solve17<T> S;
  for (;;) {
    if (tid == 0) s_next = atomicAdd(A.work, 1);
    __syncthreads();
    const int s = s_next;
    __syncthreads();
    if (s >= A.B) return;
    const size_t b0 = (size_t)s * N3;
    S.load(A, s, reinterpret_cast<T*>(tail_smem));
    const double* Fx = A.Fx + b0;
    const double* Fy = A.Fy + b0;
    const double* Fz = A.Fz + b0;
    const double* D = A.D + b0;
    // column z-march of k_residual_z (APPLY: k_apply_dot_z) over v; fn(index, value) stores;
    // partials of r~^2 (p.q) into part
    auto zmarch = [&](bool apply, const double* g, auto v, auto store) {
      double acc = 0.0;
      const int y = tid / N, x = tid - y * N;
      const bool col = tid < N2, in = col && x > 0 && y > 0 && x < N - 1 && y < N - 1;
      if (in) {
        double pm = v(tid), pc = v(tid + N2), kzm = Fz[tid];
        static_assert((N - 2) % 3 == 0, "planes in threes");
        for (int z = 1; z <= N - 2; z += 3) {  // the loads of three planes, then their sums and stores
          double pp[3], kzp[3], w[3][4], f[3][4], d[3], gg[3], r[3];
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            const int t = tid + (z + k) * N2;
            pp[k] = v(t + N2);
            kzp[k] = Fz[t];
            f[k][0] = Fx[t - 1];
            f[k][1] = Fx[t];
            f[k][2] = Fy[t - N];
            f[k][3] = Fy[t];
            w[k][0] = v(t - 1);
            w[k][1] = v(t + 1);
            w[k][2] = v(t - N);
            w[k][3] = v(t + N);
            d[k] = D[t];
            gg[k] = apply ? 0.0 : g[t];
          }
#pragma unroll
          for (int k = 0; k < 3; ++k) {
            if (apply) {
              r[k] = d[k] * pc;
#pragma unroll
              for (int q = 0; q < 4; ++q) r[k] = fma(-f[k][q], w[k][q], r[k]);
              r[k] = fma(-kzm, pm, r[k]);
              r[k] = fma(-kzp[k], pp[k], r[k]);
              acc = fma(pc, r[k], acc);
            } else {
              r[k] = fma(-d[k], pc, gg[k]);
#pragma unroll
              for (int q = 0; q < 4; ++q) r[k] = fma(f[k][q], w[k][q], r[k]);
              r[k] = fma(kzm, pm, r[k]);
              r[k] = fma(kzp[k], pp[k], r[k]);
              acc += r[k] * r[k];
            }
            pm = pc;
            pc = pp[k];
            kzm = kzp[k];
          }
#pragma unroll
          for (int k = 0; k < 3; ++k) store(tid + (z + k) * N2, r[k]);
        }
      } else if (col) {
        for (int z = 1; z <= N - 2; ++z) store(tid + z * N2, 0.0);
      }
      if (col) {
        store(tid, 0.0);
        store(tid + (N - 1) * N2, 0.0);
      }
      const double bs = group_sum<4>(acc, warp_part);
      if ((tid & 127) == 0 && (tid >> 7) < VB) part[tid >> 7] = bs;
    };
    // The per-sample scalars live in shared memory and are formed by thread 0 (an FP64 division
    // by every warp would take the FP64 pipe a tenth of a cycle).
    const double g2 = A.g2[s];
    if (tid == 0) {
      rel = 0.0;
      cyc = act = 0;
    }
    // convergence test of r~^2 = the sum of `count` partials after `inc` cycles: goes on?
    auto test = [&](int count, int inc) {
      __syncthreads();
      if (tid < 32) {
        const double t = warp_sum_partials(part, count);
        if (tid == 0) act = cta_norm_update(t, g2, A.rtol, A.maxc, inc, &rel, &cyc);
      }
      __syncthreads();
      return act != 0;
    };
    // fn(sum of `count` partials), in every thread
    auto scalar = [&](const double* p, int count, auto fn) {
      __syncthreads();
      if (tid < 32) {
        const double t = warp_sum_partials(p, count);
        if (tid == 0) bcast[0] = fn(t);
      }
      __syncthreads();
      return bcast[0];
    };
    auto none = [](int, double) {};
    if (!MIX && A.mode == kCtaStationary) {
      const double* g = A.g64 + b0;
      const double* x0 = A.x + b0;
      for (int i = tid; i < N3; i += kTailThreads) {
        S.a.g[i] = (T)g[i];
        S.a.u[i] = (T)x0[i];
      }
      __syncthreads();
      auto u = [&](int i) { return (double)S.a.u[i]; };
      for (int inc = 0;; inc = 1) {
        // k_solve_cta's test: the red residuals let a sample go on, the full one stops it
        if (inc > 0) {
          const double b = A.rtol > 0.0 ? group_sum<kTailThreads / 32>(S.red_residual(false), warp_part) : 0.0;
          if (tid == 0) {
            go_on = cyc + 1 < A.maxc && (A.rtol <= 0.0 || (g2 > 0.0 && sqrt(b / g2) > red_limit(A.rtol, false)));
            if (go_on) ++cyc;
          }
          __syncthreads();
        }
        if (inc == 0 || !go_on) {
          zmarch(false, g, u, none);
          if (!test(VB, inc)) break;
        }
        S.cycle(A, s, false);
      }
      for (int i = tid; i < N3; i += kTailThreads) A.x[b0 + i] = (double)S.a.u[i];
    } else if (MIX && A.mode == kCtaRefinement) {
      double* x = A.x + b0;
      auto xv = [&](int i) { return x[i]; };
      for (int inc = 0;; inc = 1) {
        zmarch(false, A.g64 + b0, xv, [&](int i, double r) { S.a.g[i] = (T)r; });
        if (!test(VB, inc)) break;
        S.cycle(A, s, true);
        for (int i = tid; i < N3; i += kTailThreads) x[i] += widen((float)S.a.u[i]);
        __syncthreads();
      }
    } else if (A.mode == kCtaCG) {
      double *x = A.x + b0, *R = A.R + b0, *P = A.P + b0, *Q = A.Q + b0;
      const unsigned chunk = ((unsigned)N3 + A.NB - 1) / A.NB;  // NB = 2 chunks of 256 threads' partials
      const unsigned grp = tid >> 8, lo = grp * chunk, hi = min(lo + chunk, (unsigned)N3);
      auto z = [&](unsigned i) { return widen(S.a.u[i]); };
      auto precondition = [&]() {
        S.cycle(A, s, true);
        double acc = 0.0;
        for (unsigned i = lo + (tid & 255); i < hi; i += 256) acc = fma(R[i], z(i), acc);
        const double b = group_sum<8>(acc, warp_part);
        if ((tid & 255) == 0) part[grp] = b;
      };
      auto same = [](double t) { return t; };
      double rz = 0.0, rzo = 0.0;
      zmarch(false, A.g64 + b0, [&](int i) { return x[i]; }, [&](int i, double r) { R[i] = r; });
      if (test(VB, 0)) {
        for (int i = tid; i < N3; i += kTailThreads) S.a.g[i] = (T)R[i];
        __syncthreads();
        precondition();
        rz = scalar(part, A.NB, same);
        for (int i = tid; i < N3; i += kTailThreads) P[i] = z(i);
        __syncthreads();
        for (;;) {
          zmarch(true, nullptr, [&](int i) { return P[i]; }, [&](int i, double q) { Q[i] = q; });
          const double alpha = scalar(part, VB, [&](double pq) { return pq != 0.0 ? rz / pq : 0.0; });
          double rr = 0.0, rzp = 0.0;
          for (unsigned i = lo + (tid & 255); i < hi; i += 256) {
            x[i] = fma(alpha, P[i], x[i]);
            const double rn = fma(-alpha, Q[i], R[i]);
            R[i] = rn;
            S.a.g[i] = (T)rn;
            rr = fma(rn, rn, rr);
            rzp = fma(rn, z(i), rzp);
          }
          const double s1 = group_sum<8>(rr, warp_part);
          const double s2 = group_sum<8>(rzp, warp_part);
          if ((tid & 255) == 0) {
            part[grp] = s1;
            part2[grp] = s2;
          }
          rzo = scalar(part2, A.NB, same);
          if (!test(A.NB, 1)) break;
          precondition();
          const double beta = scalar(part, A.NB, [&](double t) {
            bcast[1] = t;
            return rz != 0.0 ? (t - rzo) / rz : 0.0;
          });
          rz = bcast[1];
          for (int i = tid; i < N3; i += kTailThreads) P[i] = fma(beta, P[i], z(i));
          __syncthreads();
        }
      }
    }
    if (tid == 0) {
      A.relres[s] = rel;
      A.cycles[s] = cyc;
      A.active[s] = act;
    }
    __syncthreads();
  }
}

template <typename T>
int solve_impl(const MGSolveArgs& a, void* ws, cudaStream_t st, int* cycles_host, double* relres_host,
               int* n_unconv, int* cycles_dev, double* relres_dev) {
  const bool mixed = a.cfg.precision == MLMC_PREC_MIXED;
  const bool cg = a.cfg.accel == MLMC_ACCEL_CG;
  const bool fmg = a.cfg.accel == MLMC_ACCEL_FMG;
  Hier<T> H;
  Carver c(ws);
  layout<T>(H, c, a.B, a.n, mixed, cg);
  H.p1 = a.cfg.disc == MLMC_DISC_FE;
  H.tail_finest = fmg && a.cfg.engine != MLMC_ENGINE_BATCHED;
  const int B = a.B;
  const double W = (double)sizeof(T);
  // the sweep count of the cycle (tuned for the finest grid, or as given) and whether the
  // FP32 hierarchy runs on colour-split storage (the finest grid's smoother decides for
  // every grid)
  int nu1 = a.cfg.nu1, nu2 = a.cfg.nu2;
  // the small-grid engine: one persistent launch for the whole solve (grids up to 33^3)
  const bool use_cta = cta_engine_chosen(a.cfg, a.n, a.B);
  int sm0 = a.cfg.smoother;
  {
    resolve_tuning(a.n, a.cfg.precision, &sm0, &nu1, &nu2);
    // FP32 correction cycles on finite volumes (mixed), or FP64 stationary and FMG cycles
    // on finite volumes or P1 elements (the split kernels are instantiated for n = 5 .. 1025)
    // (not the 5^3 grid alone: it keeps the plain faces of its dense solve, nothing to sweep; not an
    // FP32 cycle without post-smoothing of more samples than half a launch's z extent, which its
    // interpolation to both colours takes twice over: the plain storage gives the same iterates)
    H.split = !use_cta && sm0 == MLMC_SMOOTH_SPLIT && a.n <= 1025 && a.n > 5 &&
              (mixed ? a.cfg.disc == MLMC_DISC_FV && (nu2 > 0 || a.B <= 32767) : !cg);
  }
  // operators of every level (k injected from k0); colour-split grids need no faces
  // except on the coarsest grid (its dense solve)
  int stride = a.st0;
  for (int j = 0; j < H.L; ++j) {
    Level<T>& v = H.lv[j];
    const dim3 gb = plane_grid(v.n * v.n, (long long)B * v.n);
    if (H.split) {
      if (j > 0) MLMC_CUDA_TRY(cudaMemsetAsync(v.g, 0, (size_t)B * split_elems(v.n) * sizeof(T), st));
      if (j < H.L - 1) {
        if constexpr (sizeof(T) == 8) {
          // FP64: stored faces, D and 1/D in the split storage (the coarsest grid keeps the
          // plain faces its dense factorisation reads)
          if (a.cfg.disc == MLMC_DISC_FE) {
            MLMC_LAUNCH("faces_fe", B * (double)v.n3 * (8.0 + 3 * W), B * (double)v.n3 * 36.0, st,
                        (k_faces_fe<double><<<gb, kPlaneThreads, 0, st>>>(a.k0, a.n_k0, stride, v.n, B,
                                                                          (double*)(void*)v.Kx, (double*)(void*)v.Ky,
                                                                          (double*)(void*)v.Kz, 1)));
          } else {
            MLMC_LAUNCH(Names<T>::faces, B * (double)v.n3 * (8.0 + 3 * W), B * (double)v.n3 * 12.0, st,
                        (k_faces_split<<<gb, kPlaneThreads, 0, st>>>(a.k0, a.n_k0, stride, v.n, B, (double*)v.Kx,
                                                                      (double*)v.Ky, (double*)v.Kz)));
          }
          MLMC_LAUNCH(Names<T>::diag, B * (double)v.n3 * 5 * W, B * (double)v.n3 * 6.0, st,
                      (k_diag_split<<<gb, kPlaneThreads, 0, st>>>(v.n, B, (const double*)v.Kx, (const double*)v.Ky,
                                                                   (const double*)v.Kz, (double*)v.D,
                                                                   (double*)v.Dinv)));
        }
        stride *= 2;
        continue;
      }
    }
    if (a.cfg.disc == MLMC_DISC_FE)
      MLMC_LAUNCH("faces_fe", B * (double)v.n3 * (8.0 + 3 * W), B * (double)v.n3 * 36.0, st,
                  (k_faces_fe<T><<<gb, kPlaneThreads, 0, st>>>(a.k0, a.n_k0, stride, v.n, B, v.Kx, v.Ky, v.Kz)));
    else
      MLMC_LAUNCH(Names<T>::faces, B * (double)v.n3 * (8.0 + 3 * W), B * (double)v.n3 * 12.0, st,
                  (k_faces<T><<<gb, kPlaneThreads, 0, st>>>(a.k0, a.n_k0, stride, v.n, B, v.Kx, v.Ky, v.Kz)));
    MLMC_LAUNCH(Names<T>::diag, B * (double)v.n3 * 5 * W, B * (double)v.n3 * 6.0, st,
                (k_diag<T, T><<<gb, kPlaneThreads, 0, st>>>(v.n, B, v.Kx, v.Ky, v.Kz, v.D, v.Dinv)));
    // restriction writes only interior coarse nodes: the boundary of g stays zero
    if (j > 0 && !H.split) MLMC_CUDA_TRY(cudaMemsetAsync(v.g, 0, (size_t)B * v.n3 * sizeof(T), st));
    stride *= 2;
  }
  // smoother per level (explicit choice, or the tuned / default one for that grid)
  for (int j = 0; j < H.L; ++j) {
    Level<T>& v = H.lv[j];
    // grids whose cycles start from a zero guess: the passes write interior nodes only
    if (j > 0 || mixed || cg)
      MLMC_CUDA_TRY(cudaMemsetAsync(v.u, 0, (size_t)B * (H.split ? split_elems(v.n) : v.n3) * sizeof(T), st));
    if (H.split) {
      H.nodal[j] = H.fused[j] = false;
      if (mixed && j < H.L - 1)
        MLMC_LAUNCH("nodal_k", B * (double)v.n3 * (8.0 + W), 0.0, st,
                    (k_nodal_k_split<<<plane_grid(v.n * v.n, (long long)B * v.n), kPlaneThreads, 0, st>>>(
                        a.k0, a.n_k0, a.st0 << j, v.n, B, (float*)(void*)v.kn)));
      continue;
    }
    int sm = a.cfg.smoother, d1 = 1, d2 = 1;
    resolve_tuning(v.n, a.cfg.precision, &sm, &d1, &d2);
    // split storage only for the whole hierarchy; where the finest grid's choice was that, every
    // grid takes its arithmetic
    if (sm == MLMC_SMOOTH_SPLIT || sm0 == MLMC_SMOOTH_SPLIT) sm = MLMC_SMOOTH_NODAL;
    // the small-grid engine runs the two-pass arithmetic (bit for bit that of the fused and
    // bulk sweeps) or the nodal one
    if (use_cta && sm != MLMC_SMOOTH_NODAL) sm = MLMC_SMOOTH_TWO_PASS;
    // the nodal-coefficient sweep exists for FP32 grids (an FP64 solve takes the two-pass)
    H.nodal[j] = v.kn != nullptr && sm == MLMC_SMOOTH_NODAL;
    H.fused[j] = v.u2 != nullptr && sm != MLMC_SMOOTH_TWO_PASS && sm != MLMC_SMOOTH_NODAL;
    if (H.nodal[j]) {
      MLMC_LAUNCH("nodal_k", B * (double)v.n3 * (8.0 + W), 0.0, st,
                  (k_nodal_k<T><<<plane_grid(v.n * v.n, (long long)B * v.n), kPlaneThreads, 0, st>>>(
                      a.k0, a.n_k0, a.st0 << j, v.n, B, v.kn)));
    }
    switch (sm) {
      case MLMC_SMOOTH_FUSED_32x16: H.tile[j] = kTile32x16; break;
      case MLMC_SMOOTH_FUSED_64x8: H.tile[j] = kTile64x8; break;
      case MLMC_SMOOTH_BULK_32x8: H.tile[j] = kBulk32x8; break;
      case MLMC_SMOOTH_BULK_32x16: H.tile[j] = kBulk32x16; break;
      case MLMC_SMOOTH_BULK_64x8: H.tile[j] = kBulk64x8; break;
      default: H.tile[j] = kTile32x8;
    }
    if (v.u2) MLMC_CUDA_TRY(cudaMemsetAsync(v.u2, 0, (size_t)B * v.n3 * sizeof(T), st));
    if (H.fused[j]) MLMC_TRY(rbgs_fused_configure<T>(H.tile[j]));
  }
  // The V-cycle as a CUDA graph: captured on the first cycle, replayed on the others.
  // Only when no per-launch events are recorded, the stream can be captured (not the
  // legacy default stream), and every level's double buffer returns to its starting
  // pointer after a cycle (nu1 + nu2 even).
  GraphRunner<T> gr;
  gr.enabled = !prof::timing_enabled() && st != nullptr && ((nu1 + nu2) % 2 == 0) && graphs_allowed();
  Level<T>& l0 = H.lv[0];
  const unsigned g0 = blocks_for((size_t)B * l0.n3, kThreads);
  H.n_act = B;
  if (mixed) {
    // the outer FP64 operator: faces of the FP64 nodal k (not of its FP32 rounding), so
    // that the refinement converges to the FP64 solution
    const dim3 gb0 = plane_grid(l0.n * l0.n, (long long)B * l0.n);
    MLMC_LAUNCH("faces64_mixed", B * (double)l0.n3 * (8.0 + 3 * 8.0), B * (double)l0.n3 * 12.0, st,
                (k_faces<double><<<gb0, kPlaneThreads, 0, st>>>(a.k0, a.n_k0, a.st0, l0.n, B, H.K64x, H.K64y,
                                                               H.K64z)));
    MLMC_LAUNCH("diag64_mixed", B * (double)l0.n3 * (3 * 8.0 + 8), B * (double)l0.n3 * 5.0, st,
                (k_diag<double, double><<<gb0, kPlaneThreads, 0, st>>>(l0.n, B, H.K64x, H.K64y, H.K64z, H.D64,
                                                                      nullptr)));
  }
  Level<T>& lc = H.lv[H.L - 1];
  MLMC_LAUNCH("coarse_setup", B * 2 * 729.0 * 8, B * 40000.0, st,
              (k_coarse_setup<T><<<(B + kCoarseWarps - 1) / kCoarseWarps, 32 * kCoarseWarps, 0, st>>>(
                  B, lc.Kx, lc.Ky, lc.Kz, H.Ainv)));
  const double h = 1.0 / (double)(a.n - 1);
  MLMC_LAUNCH("prepare", B * (double)l0.n3 * (a.f ? 16.0 : 8.0), B * (double)l0.n3, st,
              (k_prepare<<<plane_grid(a.n * a.n, (long long)B * a.n), kPlaneThreads, 0, st>>>(a.n, B, h * h, a.f,
                                                                                             H.g64, a.u)));
  if (!mixed && !cg && H.split) {
    // colour-split copies of g = h^2 f and of the initial guess; copied back at the end
    const dim3 pg0 = plane_grid(a.n * a.n, (long long)B * a.n);
    MLMC_LAUNCH("split_copy", B * (double)l0.n3 * 16.0, 0.0, st,
                (k_split_copy<double, true><<<pg0, kPlaneThreads, 0, st>>>(a.n, B, H.g64, (double*)(void*)l0.g)));
    MLMC_LAUNCH("split_copy", B * (double)l0.n3 * 16.0, 0.0, st,
                (k_split_copy<double, true><<<pg0, kPlaneThreads, 0, st>>>(a.n, B, a.u, (double*)(void*)l0.u)));
  } else if (!mixed && !cg) {
    l0.g = (T*)H.g64;
    // iterate in the workspace copy; copied back after the last cycle
    MLMC_CUDA_TRY(cudaMemcpyAsync(l0.u, a.u, (size_t)B * l0.n3 * sizeof(double), cudaMemcpyDeviceToDevice, st));
  }
  if (!mixed && cg) l0.g = (T*)H.R;  // FP64 CG: the cycle maps R to z (level-0 u)
  dim3 rg(H.NB, B);
  const unsigned sb = (B + 3) / 4;  // 128-thread blocks, one warp per sample
  MLMC_LAUNCH("norm", B * (double)l0.n3 * 8, B * (double)l0.n3 * 2, st,
              (k_sumsq<<<rg, kThreads, 0, st>>>(a.n, H.g64, H.partial)));
  MLMC_LAUNCH("norm_update", B * H.NB * 8.0, B * H.NB * 1.0, st,
              (k_norm_update<<<sb, 128, 0, st>>>(B, H.NB, H.partial, H.g2, nullptr, nullptr, nullptr, 0, 0, 0.0, 0,
                                                 nullptr)));
  MLMC_CUDA_TRY(cudaMemsetAsync(H.cycles, 0, B * sizeof(int), st));
  MLMC_CUDA_TRY(cudaMemsetAsync(H.err, 0, sizeof(int), st));
  {
    // every sample starts active; the first residual decides
    std::vector<int> ones(B, 1);
    MLMC_CUDA_TRY(cudaMemcpyAsync(H.active, ones.data(), B * sizeof(int), cudaMemcpyHostToDevice, st));
    MLMC_CUDA_TRY(cudaStreamSynchronize(st));
  }
  const double rtol = a.cfg.rtol;
  const int maxc = a.cfg.max_cycles;
  int zs = 0;
  const dim3 rz = zmarch_grid(a.n, B, &zs);
  // FP64 stationary cycles: the full residual of the samples that `mask` names (all active
  // ones), its norm and the samples that go on, added to n_active[0]
  auto full_check = [&](int inc, int* mask, int count) {
    const double Ba = (double)count;
    const int* on = mask ? mask : H.active;
    if (H.split)
      MLMC_LAUNCH("residual_norm_f64", Ba * interior(a.n) * 6.0 * 8, Ba * interior(a.n) * 16.0, st,
                  (k_residual_norm_split<<<rz, 128, 0, st>>>(a.n, zs, (const double*)l0.Kx, (const double*)l0.Ky,
                                                             (const double*)l0.Kz, (const double*)l0.D,
                                                             (const double*)l0.g, (const double*)l0.u, H.partial, on)));
    else
      MLMC_LAUNCH("residual_norm_f64", Ba * interior(a.n) * 6.0 * 8, Ba * interior(a.n) * 16.0, st,
                  (k_residual_z<T, T, T, T><<<rz, 128, 0, st>>>(a.n, zs, l0.Kx, l0.Ky, l0.Kz, l0.D, l0.g, l0.u,
                                                                nullptr, H.partial, on)));
    MLMC_LAUNCH("norm_update", B * H.NBz * 8.0, B * H.NBz * 1.0, st,
                (k_norm_update<<<sb, 128, 0, st>>>(B, H.NBz, H.partial, H.g2, H.relres, H.cycles, H.active, 1, inc,
                                                   rtol, maxc, H.n_active, mask)));
  };
  // FP64 stationary cycles on colour-split storage take the cycle's first red pass outside the
  // cycle: with the convergence test of the cycle before (k_rbgs_norm_split), or on its own for
  // the samples that `mask` names. Its replaced values go to the finest grid's spare iterate.
  const bool red_first = !mixed && !cg && !fmg && H.split && nu1 > 0 && red_fused(rtol, a.n);
  auto red_pass = [&](const int* mask, int count) {
    if constexpr (sizeof(T) == 8) {
      const dim3 gp((unsigned)(((a.n - 2) * split_groups(a.n, 4) + 127) / 128), (unsigned)(a.n - 2), (unsigned)B);
      MLMC_LAUNCH(prof::sized("rbgs_split_f64", a.n), (double)count * interior(a.n) * 3.5 * W,
                  (double)count * interior(a.n) * 0.5 * 13.0, st,
                  MLMC_SPLIT_DISPATCH(a.n, (k_rbgs_split64<LG><<<gp, 128, 0, st>>>(0, l0.Kx, l0.Ky, l0.Kz, l0.Dinv,
                                                                                 l0.g, l0.u, mask))));
    }
  };
  // Convergence test after `inc` cycles; returns the samples that go on. After an FP64 cycle
  // that ends on a black pass the red residuals decide for the samples that go on (half the FP64
  // work), the full residual for those that seem done, so reported residuals are those of a full
  // test, and so are cycle counts (red_limit says how far that holds). On colour-split storage the red residuals come with the
  // next cycle's first red pass. A 129^3 / 65^3 level of 24 samples: 75.6 ms with full tests, 66.0
  // on the red residuals; later 54.8 -> 52.5 with the pass and its test in one (6.3 ms of tests,
  // 3.3 of them the pass); 65^3 x 19 6.72 -> 6.47.
  auto residual_check = [&](int inc) -> int {
    MLMC_CUDA_TRY(cudaMemsetAsync(H.n_active, 0, 2 * sizeof(int), st));
    const double Ba = (double)H.n_act;
    int na[2] = {0, 0};
    if (mixed) {
      if (H.split)
        MLMC_LAUNCH("residual_mixed", Ba * interior(a.n) * (3 * 8.0 + 8 * 3 + W), Ba * interior(a.n) * 16.0, st,
                    (k_residual_z<double, double, double, T, true><<<rz, 128, 0, st>>>(
                        a.n, zs, H.K64x, H.K64y, H.K64z, H.D64, H.g64, a.u, l0.g, H.partial, H.active)));
      else
        MLMC_LAUNCH("residual_mixed", Ba * interior(a.n) * (3 * 8.0 + 8 * 3 + W), Ba * interior(a.n) * 16.0, st,
                    (k_residual_z<double, double, double, T><<<rz, 128, 0, st>>>(a.n, zs, H.K64x, H.K64y, H.K64z,
                                                                                 H.D64, H.g64, a.u, l0.g, H.partial,
                                                                                 H.active)));
      MLMC_LAUNCH("norm_update", B * H.NBz * 8.0, B * H.NBz * 1.0, st,
                  (k_norm_update<<<sb, 128, 0, st>>>(B, H.NBz, H.partial, H.g2, H.relres, H.cycles, H.active, 1, inc,
                                                     rtol, maxc, H.n_active)));
    } else if (inc > 0 && nu1 + nu2 > 0 && H.L > 1) {
      const bool fused = red_first;
      const int slots = fused ? (a.n - 2) * split_groups(a.n, 4) : (a.n - 2) * ((a.n - 1) / 2);
      const dim3 rr((unsigned)((slots + 127) / 128), rz.y, (unsigned)B);
      const int NBr = (int)(rr.x * rr.y);
      if (H.split && !fused) {  // no pre-smoothing, or a tolerance below red_fused's: the full residual
        full_check(inc, nullptr, H.n_act);
        MLMC_CUDA_TRY(cudaMemcpyAsync(na, H.n_active, sizeof(na), cudaMemcpyDeviceToHost, st));
        MLMC_CUDA_TRY(cudaStreamSynchronize(st));
        return H.n_act = na[0];
      }
      if constexpr (sizeof(T) == 8) {
        if (fused)
          MLMC_LAUNCH("rbgs_norm_f64", Ba * interior(a.n) * 4.5 * 8, Ba * interior(a.n) * 8.5, st,
                      MLMC_SPLIT_DISPATCH(a.n, (k_rbgs_norm_split<LG><<<rr, 128, 0, st>>>(
                                                   zs, l0.Kx, l0.Ky, l0.Kz, l0.D, l0.Dinv, l0.g, l0.u, l0.u2,
                                                   H.partial, H.active))));
      }
      if (!fused)
        MLMC_LAUNCH("residual_norm_red", Ba * interior(a.n) * 4.0 * 8, Ba * interior(a.n) * 8.0, st,
                    (k_norm_red_z<T><<<rr, 128, 0, st>>>(a.n, zs, l0.Kx, l0.Ky, l0.Kz, l0.D, l0.g, l0.u, H.partial,
                                                         H.active)));
      MLMC_LAUNCH("norm_update", B * NBr * 8.0, B * NBr * 1.0, st,
                  (k_norm_red<<<sb, 128, 0, st>>>(B, NBr, H.partial, H.g2, H.cycles, H.active, H.cand, inc,
                                                  red_limit(rtol, fused), maxc, H.n_active)));
      MLMC_CUDA_TRY(cudaMemcpyAsync(na, H.n_active, sizeof(na), cudaMemcpyDeviceToHost, st));
      MLMC_CUDA_TRY(cudaStreamSynchronize(st));
      if (na[1] == 0) return H.n_act = na[0];
      if constexpr (sizeof(T) == 8) {
        if (fused) {
          const dim3 gp((unsigned)((slots + 127) / 128), (unsigned)(a.n - 2), (unsigned)B);
          MLMC_LAUNCH("restore_red", (double)na[1] * interior(a.n) * 8.0, 0.0, st,
                      MLMC_SPLIT_DISPATCH(a.n, (k_restore_red<LG><<<gp, 128, 0, st>>>(l0.u2, l0.u, H.cand))));
        }
      }
      const int on = na[0];
      full_check(0, H.cand, na[1]);
      MLMC_CUDA_TRY(cudaMemcpyAsync(na, H.n_active, sizeof(na), cudaMemcpyDeviceToHost, st));
      MLMC_CUDA_TRY(cudaStreamSynchronize(st));
      if (fused && na[0] > on) red_pass(H.cand, na[0] - on);  // candidates that go on after all
      return H.n_act = na[0];
    } else {
      full_check(inc, nullptr, H.n_act);
    }
    MLMC_CUDA_TRY(cudaMemcpyAsync(na, H.n_active, sizeof(na), cudaMemcpyDeviceToHost, st));
    MLMC_CUDA_TRY(cudaStreamSynchronize(st));
    return H.n_act = na[0];
  };
  if (use_cta) {
    CtaArgs<T> A;
    A.L = H.L;
    A.B = B;
    A.nu1 = nu1;
    A.nu2 = nu2;
    A.maxc = maxc;
    A.rtol = rtol;
    A.red_limit = red_limit(rtol, true);
    A.red_fused = red_fused(rtol, a.n);
    A.mode = cg ? kCtaCG : (mixed ? kCtaRefinement : kCtaStationary);
    for (int j = 0; j < H.L; ++j) {
      Level<T>& v = H.lv[j];
      A.lv[j].n = v.n;
      A.lv[j].Kx = v.Kx;
      A.lv[j].Ky = v.Ky;
      A.lv[j].Kz = v.Kz;
      A.lv[j].D = v.D;
      A.lv[j].Dinv = v.Dinv;
      A.lv[j].kn = H.nodal[j] ? v.kn : nullptr;
      A.lv[j].u = v.u;
      A.lv[j].g = v.g;
      A.lv[j].r = v.r;
    }
    A.Ainv = H.Ainv;
    A.Fx = mixed ? H.K64x : (const double*)(const void*)l0.Kx;
    A.Fy = mixed ? H.K64y : (const double*)(const void*)l0.Ky;
    A.Fz = mixed ? H.K64z : (const double*)(const void*)l0.Kz;
    A.D = mixed ? H.D64 : (const double*)(const void*)l0.D;
    A.g64 = H.g64;
    A.x = (!mixed && !cg) ? (double*)(void*)l0.u : a.u;
    A.R = H.R;
    A.P = H.P;
    A.Q = H.Q;
    A.Z = H.Z;
    A.g2 = H.g2;
    A.relres = H.relres;
    A.cycles = H.cycles;
    A.active = H.active;
    A.work = H.n_active;
    A.NB = H.NB;
    A.slabs = apply_slabs(a.n, &A.zslab);
    int dev = 0, sms = 0, per_sm = 0;
    MLMC_CUDA_TRY(cudaGetDevice(&dev));
    MLMC_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    MLMC_CUDA_TRY(cudaMemsetAsync(H.n_active, 0, sizeof(int), st));
    // k_solve17 fills an SM with one sample: always the faster form for FP32 cycles (17^3 x 400
    // mixed refinement: 1.02 ms against 1.57), for FP64 ones while every SM has at most one sample
    // (one sample 0.51 ms against 0.84; 4096 of them 15.1 against 14.2 when both were measured,
    // k_solve_cta 11.8 since: its four samples per SM fill the FP64 pipe)
    if (a.n == 17 && nu1 > 0 && nu2 > 0 && !H.nodal[0] && !H.nodal[1] && A.NB == 2 && A.slabs == 1 && (mixed || B <= sms)) {
      const size_t smem = Solve17<T>::elems * sizeof(T);
      MLMC_CUDA_TRY(allow_dynamic_smem<k_solve17<T>>(smem));
      MLMC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_solve17<T>, kTailThreads, smem));
      const int grid = B < sms * (per_sm > 0 ? per_sm : 1) ? B : sms * (per_sm > 0 ? per_sm : 1);
      MLMC_LAUNCH(prof::sized(sizeof(T) == 4 ? "solve_cta_mixed" : "solve_cta_f64", a.n), 0.0, 0.0, st,
                  (k_solve17<T><<<grid, kTailThreads, smem, st>>>(A)));
    } else {
      MLMC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_solve_cta<T>, kCtaThreads, 0));
      const int grid = B < sms * (per_sm > 0 ? per_sm : 1) ? B : sms * (per_sm > 0 ? per_sm : 1);
      MLMC_LAUNCH(prof::sized(sizeof(T) == 4 ? "solve_cta_mixed" : "solve_cta_f64", a.n), 0.0, 0.0, st,
                  (k_solve_cta<T><<<grid, kCtaThreads, 0, st>>>(A)));
    }
    MLMC_CUDA_TRY(cudaGetLastError());
  }
  if (cg && !use_cta) {
    const int st_pcg = H.split ? pcg_loop<T, true>(H, a, nu1, nu2, rtol, maxc, st, gr)
                               : pcg_loop<T, false>(H, a, nu1, nu2, rtol, maxc, st, gr);
    if (st_pcg < 0) return st_pcg;
  }
  if (fmg) {
    // One FMG cycle (nested iteration, Sec. 7): every grid's own right-hand side h_j^2 f
    // (f = 1), the exact solve on the coarsest grid, then per finer grid the P1 (or
    // trilinear) interpolation of the coarser solution and max_cycles V(nu1, nu2) cycles.
    for (int j = 1; j < H.L; ++j) {
      Level<T>& v = H.lv[j];
      const double hj = 1.0 / (double)(v.n - 1);
      if (H.split)
        MLMC_LAUNCH("prepare", B * (double)v.n3 * 8.0, B * (double)v.n3, st,
                    (k_prepare<true><<<plane_grid(v.n * v.n, (long long)B * v.n), kPlaneThreads, 0, st>>>(
                        v.n, B, hj * hj, nullptr, (double*)v.g, (double*)v.u)));
      else
        MLMC_LAUNCH("prepare", B * (double)v.n3 * 8.0, B * (double)v.n3, st,
                    (k_prepare<<<plane_grid(v.n * v.n, (long long)B * v.n), kPlaneThreads, 0, st>>>(
                        v.n, B, hj * hj, nullptr, (double*)v.g, (double*)v.u)));
    }
    vcycle(H, H.L - 1, nu1, nu2, st, true);
    for (int j = H.L - 2; j >= 0; --j) {
      Level<T>& v = H.lv[j];
      MLMC_CUDA_TRY(cudaMemsetAsync(v.u, 0, (size_t)B * (H.split ? split_elems(v.n) : v.n3) * sizeof(T), st));
      prolong_level(H, j, nu1 > 0, st);  // the cycle's first red pass overwrites the red nodes
      // with MLMC_FMG_GRAPHS=1 the cycles of grid j replay one graph captured for them (on
      // created streams): a level alone runs 4-6% faster, but the capture and instantiation
      // of every grid's graph in every solve cost more than they save while other level
      // streams keep the GPU busy, so direct launches are the default
      GraphRunner<T> fr;
      fr.enabled = gr.enabled && fmg_graphs();
      for (int cyc = 0; cyc < maxc; ++cyc) MLMC_TRY(fr.run(H, nu1, nu2, st, false, j));
    }
    std::vector<int> cyc(B, maxc);
    MLMC_CUDA_TRY(cudaMemcpyAsync(H.cycles, cyc.data(), B * sizeof(int), cudaMemcpyHostToDevice, st));
    // the final relative residual, for the statistics only (the cycle's work is fixed)
    MLMC_CUDA_TRY(cudaMemsetAsync(H.n_active, 0, sizeof(int), st));
    full_check(0, nullptr, B);
  }
  const bool cycling = !(cg || fmg || use_cta);
  if (cycling && !mixed && rtol <= 0.0) {
    // fixed FP64 cycles: nothing depends on a residual before the last one
    for (int c = 0; c < maxc; ++c) MLMC_TRY(gr.run(H, nu1, nu2, st, false));
    MLMC_CUDA_TRY(cudaMemsetAsync(H.n_active, 0, 2 * sizeof(int), st));
    full_check(maxc, nullptr, B);
  }
  int na = cycling && (mixed || rtol > 0.0) ? residual_check(0) : 0;
  if (na < 0) return na;
  bool first_cycle = true;
  while (na > 0) {
    if (mixed) {
      MLMC_CUDA_TRY(clear_guess(H, 0, nu1, st));
      MLMC_TRY(gr.run(H, nu1, nu2, st, true));
      const dim3 ug = plane_grid(a.n * a.n, (long long)B * a.n);
      if (H.split)
        MLMC_LAUNCH("update_mixed", H.n_act * (double)l0.n3 * (W + 16), H.n_act * (double)l0.n3, st,
                    (k_update_mixed<true><<<ug, kPlaneThreads, 0, st>>>(a.n, B, (const float*)H.lv[0].u, a.u,
                                                                          H.active)));
      else
        MLMC_LAUNCH("update_mixed", H.n_act * (double)l0.n3 * (W + 16), H.n_act * (double)l0.n3, st,
                    (k_update_mixed<false><<<ug, kPlaneThreads, 0, st>>>(a.n, B, (const float*)H.lv[0].u, a.u,
                                                                           H.active)));
    } else {
      if (red_first && first_cycle) red_pass(H.active, H.n_act);
      first_cycle = false;
      MLMC_TRY(gr.run(H, nu1, nu2, st, false, 0, red_first));
    }
    na = residual_check(1);
    if (na < 0) return na;
  }
  // FP64 solves iterate in place on the caller's u; the fused smoother may leave the
  // latest iterate in the spare buffer
  if (!mixed && !cg && H.split)
    MLMC_LAUNCH("split_copy", B * (double)l0.n3 * 16.0, 0.0, st,
                (k_split_copy<double, false><<<plane_grid(a.n * a.n, (long long)B * a.n), kPlaneThreads, 0, st>>>(
                    a.n, B, (const double*)(const void*)H.lv[0].u, a.u)));
  else if (!mixed && !cg)
    MLMC_CUDA_TRY(cudaMemcpyAsync(a.u, H.lv[0].u, (size_t)B * l0.n3 * sizeof(double), cudaMemcpyDeviceToDevice, st));
  MLMC_CUDA_TRY(cudaGetLastError());
  if (cycles_dev)
    MLMC_CUDA_TRY(cudaMemcpyAsync(cycles_dev, H.cycles, B * sizeof(int), cudaMemcpyDeviceToDevice, st));
  if (relres_dev)
    MLMC_CUDA_TRY(cudaMemcpyAsync(relres_dev, H.relres, B * sizeof(double), cudaMemcpyDeviceToDevice, st));
  std::vector<int> cyc(B);
  std::vector<double> rel(B);
  int errw = 0;
  MLMC_CUDA_TRY(cudaMemcpyAsync(&errw, H.err, sizeof(int), cudaMemcpyDeviceToHost, st));
  MLMC_CUDA_TRY(cudaMemcpyAsync(cyc.data(), H.cycles, B * sizeof(int), cudaMemcpyDeviceToHost, st));
  MLMC_CUDA_TRY(cudaMemcpyAsync(rel.data(), H.relres, B * sizeof(double), cudaMemcpyDeviceToHost, st));
  MLMC_CUDA_TRY(cudaStreamSynchronize(st));
  if (errw == 1) {
    set_error("a staging wait of the fused smoother ran out of its time budget");
    return MLMC_ERR_TIMEOUT;
  }
  if (errw) {
    set_error("the fused smoother's bounds check failed (code %d)", errw);
    return MLMC_ERR_CUDA;
  }
  int bad = 0;
  for (int s = 0; s < B; ++s) {
    if (cycles_host) cycles_host[s] = cyc[s];
    if (relres_host) relres_host[s] = rel[s];
    if (!fmg && rtol > 0.0 && !(rel[s] <= rtol)) ++bad;
  }
  if (n_unconv) *n_unconv = bad;
  return MLMC_OK;
}

}  // namespace

size_t mg_workspace_bytes(int B, int n, int precision, int accel) {
  Carver c(nullptr);
  if (precision == MLMC_PREC_MIXED) {
    Hier<float> H;
    layout<float>(H, c, B, n, true, accel == MLMC_ACCEL_CG);
  } else {
    Hier<double> H;
    layout<double>(H, c, B, n, false, accel == MLMC_ACCEL_CG);
  }
  return c.off;
}

int mg_solve_dev(const MGSolveArgs& a, void* ws, cudaStream_t st, int* cycles_host, double* relres_host,
                 int* n_unconv, int* cycles_dev, double* relres_dev) {
  if (a.cfg.precision == MLMC_PREC_MIXED)
    return solve_impl<float>(a, ws, st, cycles_host, relres_host, n_unconv, cycles_dev, relres_dev);
  return solve_impl<double>(a, ws, st, cycles_host, relres_host, n_unconv, cycles_dev, relres_dev);
}

int interpolate_dev(const double* uc, int nf, int B, double* uf, cudaStream_t st) {
  MLMC_CUDA_TRY(cudaMemsetAsync(uf, 0, (size_t)B * cube(nf) * sizeof(double), st));
  const int mc = (nf + 1) / 2 - 1;
  MLMC_LAUNCH("interpolate_f64", B * (2.0 * (double)cube(nf) + (double)cube((nf + 1) / 2)) * 8.0,
              B * interior(nf) * 4.375, st,
              (k_prolong_blk<double><<<plane_grid(mc * mc, (long long)B * mc), 128, 0, st>>>(nf, B, uc, uf,
                                                                                             nullptr)));
  return MLMC_OK;
}

size_t qoi_scratch_bytes(int B, int n) {
  const int S = (n - 1) / 2 + 1;
  const size_t a = (size_t)B * reduce_blocks(cube(S)) * sizeof(double);
  const size_t b = (size_t)B * reduce_blocks((size_t)(n - 1) * (n - 1)) * sizeof(double);
  return a256(a > b ? a : b);
}

int qoi_dev(const double* u, int n, int B, double* Q, void* scratch, cudaStream_t st) {
  const int S = (n - 1) / 2 + 1;
  const int NB = reduce_blocks(cube(S));
  double* partial = (double*)scratch;
  MLMC_LAUNCH("qoi", B * (double)cube(S) * 8, B * (double)cube(S) * 6, st,
              (k_qoi<<<dim3(NB, B), kThreads, 0, st>>>(n, u, partial)));
  const double h = 1.0 / (double)(n - 1);
  MLMC_LAUNCH("qoi_final", B * NB * 8.0, B * NB * 1.0, st,
              (k_qoi_final<<<(B + 127) / 128, 128, 0, st>>>(B, NB, 8.0 * h * h * h, partial, Q)));
  MLMC_CUDA_TRY(cudaGetLastError());
  return MLMC_OK;
}

int qoi_any(int qoi, const double* u, int n, int B, double* Q, void* scratch, const double* k0, int n_k0, int st0,
            cudaStream_t st) {
  if (qoi == MLMC_QOI_MEAN) return qoi_dev(u, n, B, Q, scratch, st);
  if (qoi == MLMC_QOI_POINT) {
    MLMC_LAUNCH("qoi", B * 8.0, 0.0, st, (k_qoi_point<<<(B + 127) / 128, 128, 0, st>>>(n, B, u, Q)));
    return MLMC_OK;
  }
  const int NB = reduce_blocks((size_t)(n - 1) * (n - 1));
  double* partial = (double*)scratch;
  MLMC_LAUNCH("qoi", B * (double)(n - 1) * (n - 1) * 8 * 16, B * (double)(n - 1) * (n - 1) * 6 * 8, st,
              (k_qoi_flux<<<dim3(NB, B), kThreads, 0, st>>>(n, u, k0, n_k0, st0, partial)));
  const double h = 1.0 / (double)(n - 1);
  MLMC_LAUNCH("qoi_final", B * NB * 8.0, B * NB * 1.0, st,
              (k_qoi_final<<<(B + 127) / 128, 128, 0, st>>>(B, NB, h / 6.0, partial, Q)));
  MLMC_CUDA_TRY(cudaGetLastError());
  return MLMC_OK;
}

}  // namespace mlmc
