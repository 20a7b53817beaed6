// Host run of the one-launch cycle's launcher and of the cycle runner
// (tests/test_tail_failure_host.py), their own text, with a runtime that refuses the kernel's
// dynamic shared memory: every cycle has to report it, launched directly or captured.
#include <cstddef>
#include <cstdio>
#include <shared_mutex>
#include <type_traits>
#include <vector>

typedef int cudaError_t;
typedef void* cudaStream_t;
struct Graph {
  int kernels = 0;
};
typedef Graph* cudaGraph_t;
typedef Graph* cudaGraphExec_t;
enum { cudaSuccess = 0, cudaErrorInvalidValue = 1, cudaErrorMemoryAllocation = 2, cudaStreamCaptureModeThreadLocal = 2 };
enum { MLMC_OK = 0, MLMC_ERR_OOM = -2, MLMC_ERR_CUDA = -5 };

static cudaError_t opt_in = cudaSuccess;  // what the runtime says to the shared-memory limit
static int launched = 0, graphs = 0;
static bool capturing = false;
static Graph* captured = nullptr;

static const char* cudaGetErrorString(cudaError_t) { return ""; }
static void set_error(const char*, ...) {}
#define MLMC_CUDA_TRY(expr)                                                  \
  do {                                                                       \
    const cudaError_t _e = (expr);                                           \
    if (_e != cudaSuccess) return _e == cudaErrorMemoryAllocation ? MLMC_ERR_OOM : MLMC_ERR_CUDA; \
  } while (0)
#define MLMC_LAUNCH(cls, bytes, flops, st, launch_expr) \
  do {                                                  \
    (void)(cls), (void)(bytes), (void)(flops), (void)(st); \
    launch_expr;                                        \
  } while (0)
static std::shared_mutex& capture_lock() {
  static std::shared_mutex mu;
  return mu;
}
namespace prof {
struct Tape {};
static void tape_begin() {}
static Tape tape_end() { return Tape{}; }
static void tape_replay(const Tape&, double) {}
static const char* sized(const char* s, int) { return s; }
}  // namespace prof
static cudaError_t cudaStreamBeginCapture(cudaStream_t, int) {
  capturing = true;
  captured = new Graph;
  return cudaSuccess;
}
static cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  capturing = false;
  *g = captured;
  ++graphs;
  return cudaSuccess;
}
static cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, int) {
  *e = new Graph(*g);
  return cudaSuccess;
}
static cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  delete g;
  --graphs;
  return cudaSuccess;
}
static cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
  delete e;
  return cudaSuccess;
}
static cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
  launched += e->kernels;
  return cudaSuccess;
}

#include "hier.inc"  // Level, TailLevel, TailArgs

template <typename T, int N, bool CS>
struct TailGrid {
  static constexpr int shared_iter = 2 * N * N * N + (N * N * N + 1) / 2;
};
constexpr int kTailThreads = 512;
template <typename T>
struct Hier {
  int B = 3, n_act = 3;
  Level<T> lv[3];
  double* Ainv = nullptr;
  int* active = nullptr;
  bool split = false, p1 = false, nodal[3] = {};
  cudaError_t failed = cudaSuccess;
};
static double interior(int n) { return (double)(n - 2) * (n - 2) * (n - 2); }
template <typename T, int N0, bool SPLIT, bool P1>
static void k_vcycle_tail(TailArgs<T>) {}
template <auto Kernel>
static cudaError_t allow_dynamic_smem(size_t) {
  return opt_in;
}
template <typename A>
static void emu_launch(const A&) {
  if (capturing)
    ++captured->kernels;
  else
    ++launched;
}

#include "tail.inc"  // tail_launch, vcycle_tail
template <typename T>
static void vcycle(Hier<T>& H, int j, int nu1, int nu2, cudaStream_t st, bool zero, bool) {
  vcycle_tail(H, j, nu1, nu2, st, zero);
}
#include "runner.inc"  // GraphRunner

template <typename T>
static int run(int n, bool graph, bool split, bool p1) {
  Hier<T> H;
  H.lv[0].n = n;
  H.lv[1].n = (n + 1) / 2;
  H.split = split;
  H.p1 = p1;
  int bad = 0;
  {
    GraphRunner<T> gr;
    gr.enabled = graph;
    launched = 0;
    for (int c = 0; c < 3; ++c) bad += gr.run(H, 2, 2, nullptr, true) != MLMC_OK;
    bad += launched != 3;  // the kernel ran in every cycle
  }
  opt_in = cudaErrorInvalidValue;
  for (int call = 0; call < 2; ++call) {  // a second solve is told as well
    Hier<T> G = H;
    GraphRunner<T> gr;
    gr.enabled = graph;
    launched = 0;
    for (int c = 0; c < 3; ++c) bad += gr.run(G, 2, 2, nullptr, true) != MLMC_ERR_CUDA;
    bad += launched != 0;
  }
  opt_in = cudaSuccess;
  bad += graphs != 0;
  if (bad) std::printf("n %d, graph %d, split %d, p1 %d: %d wrong\n", n, graph, split, p1, bad);
  return bad;
}

int main() {
  int bad = 0;
  for (int n : {9, 17})
    for (int graph = 0; graph < 2; ++graph)
      for (int split = 0; split < 2; ++split) {
        bad += run<double>(n, graph, split, false) + run<double>(n, graph, split, true);
        bad += run<float>(n, graph, split, false);
      }
  return bad ? 1 : 0;
}
