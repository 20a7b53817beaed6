// Tuning table (see tune.cuh).
#include <map>
#include <mutex>
#include <utility>

#include "common.cuh"
#include "tune.cuh"

namespace mlmc {
namespace {
std::mutex g_mu;
std::map<std::pair<int, int>, std::pair<int, int>> g_table;
}  // namespace

void tune_store(int n, int precision, int smoother, int nu) {
  std::lock_guard<std::mutex> lk(g_mu);
  g_table[{n, precision}] = {smoother, nu};
}

bool tune_lookup(int n, int precision, int* smoother, int* nu) {
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_table.find({n, precision});
  if (it == g_table.end()) return false;
  *smoother = it->second.first;
  *nu = it->second.second;
  return true;
}

void tune_clear() {
  std::lock_guard<std::mutex> lk(g_mu);
  g_table.clear();
}

void resolve_tuning(int n, int precision, int* smoother, int* nu1, int* nu2) {
  int ts = 0, tnu = 0;
  const bool tuned = tune_lookup(n, precision, &ts, &tnu);
  if (*smoother == MLMC_SMOOTH_AUTO) {
    // untuned grids: the colour-split storage where a row of a colour is long enough for its
    // 16-byte groups to pay for the copies into it and back, the two-pass sweep below. Measured
    // (solves; auto was two-pass): FP32 correction cycles 33^3 x 48 3.74 (two-pass 4.12) ms, 33^3 x
    // 2 1.72 (1.85), 65^3 x 20 7.07 (8.85); FP64 33^3 x 150 8.40 (8.10), 65^3 x 19 8.49 (8.72), 65^3
    // x 108 P1 / FMG level 20.3 (20.7), 129^3 level of 24 63 (68.5). Bit for bit the two-pass
    // iterates in FP64. Where the split storage does not apply the choice falls back (solve_impl).
    const int from = precision == MLMC_PREC_MIXED ? 33 : 65;
    *smoother = tuned ? ts : (n >= from ? MLMC_SMOOTH_SPLIT : MLMC_SMOOTH_TWO_PASS);
  }
  if (*nu1 == 0 && *nu2 == 0) {
    const int nu = tuned ? tnu : 2;
    *nu1 = nu;
    *nu2 = nu;
  }
}

}  // namespace mlmc
