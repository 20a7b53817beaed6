// Host run of the tcgen05 field kernel's issuing thread (tests/test_umma_drain_host.py): its own
// text, with the barriers as phase counters. An operation in flight (a bulk copy, the arrival of a
// commit) lands only when the thread waits for its barrier, so what has not been waited for when
// the thread returns is what the block could leave behind. The other threads either take part or
// have given up; any single wait of the thread may run out.
#include <algorithm>
#include <cstdint>
#include <cstdio>
#include <map>
#include <set>
using std::max;

struct Barrier {
  int phase = 0, pending = 0;  // completed phases; operations in flight that will complete the next ones
};
static std::set<Barrier*> all;
static int waits, expire;  // waits so far; the one that runs out (-1: none)
static Barrier *read_out, *sums;  // the warps arrive on the first once they have seen the second complete
constexpr long long kDrainBudget = 1LL << 40;

static void arrive_later(Barrier* b) {
  all.insert(b);
  ++b->pending;
}
static void mbar_arrive_expect_tx(Barrier*, unsigned) {}
static void bulk_g2s(void*, const void*, unsigned, Barrier* b) { arrive_later(b); }
static bool mbar_wait_bounded(Barrier* b, unsigned parity, long long budget) {
  if (budget != kDrainBudget && waits++ == expire) return false;
  while (b->pending > 0 && (b->phase & 1) == (int)parity) --b->pending, ++b->phase;
  const bool done = (b->phase & 1) != (int)parity;
  if (done && b == read_out) sums->phase += sums->pending, sums->pending = 0;
  return done;
}
static void atomicExch(int*, int) {}
static unsigned smem_addr(const void*) { return 0; }
namespace umma {
constexpr unsigned kLeadingBytes = 0, kStrideBytes = 0;
static void fence_after_sync() {}
static uint64_t smem_desc(unsigned, unsigned, unsigned) { return 0; }
static uint32_t idesc_bf16_f32(int, int) { return 0; }
static void mma_bf16(uint32_t, uint64_t, uint64_t, uint32_t, uint32_t) {}
static void commit(Barrier* b) { arrive_later(b); }
}  // namespace umma

struct S {
  static constexpr int stage = 64, a_stage = 32, b_stage = 16;
};

// operations in flight when the thread returns
template <int NS, int N, bool MULTI>
static int issue(int KS, int inject, bool others, int fail) {
  constexpr int kFoldSteps = 32, kTcSlices = 7, kUmATile = 4096, kUmM = 128;
  static unsigned char mem[NS * 64], table[1 << 12];
  unsigned char *sm = mem, *xu = table;
  Barrier bfull[NS], full[NS], empty[NS], accs, accr, nothing;
  Barrier *accf = &accs, *acce = &accr, *never = &nothing;
  if (others)  // the staging warps' arrivals, as many as the thread can wait for
    for (int q = 0; q < KS; ++q) {
      ++full[q % NS].pending;
      ++accr.pending;
    }
  const uint32_t tmem = 0;
  const long long budget = 1;
  int word = 0, *err = &word;
  all.clear();
  read_out = acce;
  sums = accf;
  waits = 0;
  expire = fail;
#include "issuer.inc"
  int left = 0;
  for (Barrier* b : all) left += b->pending;
  return left;
}

int main() {
  int runs = 0, bad_runs = 0;
  auto check = [&](const char* what, int KS, int inject, bool others, int fail, int left) {
    ++runs;
    if (!left) return;
    if (bad_runs++ < 10)
      std::printf("%s KS %d inject %d others %d wait %d: %d in flight at the end\n", what, KS, inject, others, fail, left);
  };
  for (int KS : {1, 2, 3, 4, 5, 7, 31, 32})
    for (int others = 0; others < 2; ++others)
      for (int inject = 0; inject < 2; ++inject)
        for (int fail = -1; fail < 3 * KS + 2; ++fail) {
          check("N 16", KS, inject, others, fail, issue<2, 16, false>(KS, inject, others, fail));
          check("N 32", KS, inject, others, fail, issue<3, 32, false>(KS, inject, others, fail));
          check("N 64", KS, inject, others, fail, issue<4, 64, false>(KS, inject, others, fail));
        }
  for (int KS : {33, 64, 65, 100})
    for (int others = 0; others < 2; ++others)
      for (int fail = -1; fail < 3 * KS + 8; ++fail) {
        check("N 16 folds", KS, 0, others, fail, issue<2, 16, true>(KS, 0, others, fail));
        check("N 64 folds", KS, 0, others, fail, issue<4, 64, true>(KS, 0, others, fail));
      }
  std::printf("%d of %d runs left something in flight\n", bad_runs, runs);
  return bad_runs ? 1 : 0;
}
