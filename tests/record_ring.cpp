// The record ring of the 128-token kernel on the host: fwd_sm100_records.cuh with mbarriers and TMA loads of this file,
// its roles as coroutines that a random scheduler steps from one barrier operation to the next.
//
//   record_ring SEEDS TILES...     the records in order: a number of tiles for each chunk, "/" after an item's last one
//
// Prints "ok" when every interleaving loads the tiles of the records in order and comes to its end; otherwise says
// which one stalled, or loaded something else, and exits with 1.
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
#include <ucontext.h>

#include <memory>
#include <random>
#include <string>
#include <vector>

#define __device__
#define __forceinline__ inline
struct float2 { float x, y; };
struct CUtensorMap { int id; };

namespace sol {
namespace fwd {

constexpr int kRowsQ = 128;
struct Params { long long wait_limit; int rows_inner; };

// ---- scheduler
struct Task {
  ucontext_t ctx;
  std::vector<char> stack = std::vector<char>(1 << 16);
  bool done = false;
  uint64_t* bar = nullptr;                       // waits for this barrier's phase
  uint32_t parity = 0;
};
std::vector<std::unique_ptr<Task>> tasks;
Task* current;
ucontext_t main_ctx;
bool stalled;

void yield() { swapcontext(&current->ctx, &main_ctx); }

// ---- mbarriers: low byte arrivals still missing, next byte their number, bit 16 the phase
void mbar_init(uint64_t* bar, uint32_t count) { *bar = count | count << 8; }
bool complete(uint64_t bar, uint32_t parity) { return ((bar >> 16) & 1) != parity; }
void mbar_arrive(uint64_t* bar) {
  if ((--*bar & 0xff) == 0) *bar = ((*bar ^ 0x10000) & ~0xffull) | ((*bar >> 8) & 0xff);
  yield();
}
void mbar_arrive_expect_tx(uint64_t* bar, uint32_t) { mbar_arrive(bar); }   // the copy lands at once
bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  yield();
  return complete(*bar, parity);
}
bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int*, long long) {
  if (!complete(*bar, parity)) {
    current->bar = bar;
    current->parity = parity;
    yield();
    current->bar = nullptr;
  }
  return !stalled;
}

// ---- loads: (map, row) in the order they are issued
std::vector<std::pair<int, int>> loads[3];       // Q, K side, V side
void tma_load_4d(void*, const CUtensorMap* m, uint64_t*, int c0, int c1, int c2, int c3) {
  if (c0 == 0) loads[m->id == 0 ? 0 : (m->id & 1 ? 1 : 2)].push_back({m->id, c1 + 100000 * c2 + 1000000 * c3});
}
template <class S>
void flag_abort(S& sm, const Params&, int) { sm.abort_flag = 1; }

}  // namespace fwd
}  // namespace sol

#define WAIT(bar, parity, slot) mbar_wait((bar), (parity), &sm.abort_flag, wait_limit)
#define PROF_DECL
#define PROF_COUNT(slot)
#define PROF_FLUSH(role)
#define PROF_ACC(slot) nullptr
#define PROF_T0
#define PROF_ADD(slot)
#include "fwd_sm100_records.cuh"

using namespace sol::fwd;
using C = Cfg<128, 128>;

static Shared<C> sm;
static std::vector<std::vector<int>> items;      // tiles of each chunk of each item
static const Params prm{0, 1};
static const CUtensorMap tm_q{0}, tm_k{1}, tm_v{2}, tm_kc{3}, tm_vm{4};
static const long long wait_limit = 0;

static void router() {                           // what router_role writes
  uint32_t n = 0;
  for (size_t w = 0; w < items.size(); ++w) {
    bool any = false;
    for (size_t t = 0; t < items[w].size(); ++t, ++n) {
      if (!WAIT(&sm.rec_empty[n % kRecords], ((n / kRecords) & 1) ^ 1, 0)) return;
      Record<C>& rec = sm.rec[n % kRecords];
      memset(&rec, 0xff, sizeof(rec));
      const int tiles = items[w][t];
      const bool last = t + 1 == items[w].size();
      rec.work = (int)w; rec.b = (int)w % 2; rec.h = (int)w % 3; rec.q_row = (int)w * 128;
      for (int e = 0; e < tiles; ++e) rec.desc[1 + e] = (uint32_t)((t * 128 + e) * 128) << 5;
      if (!any && tiles) rec.desc[1] |= kTileFirst;
      any |= tiles > 0;
      if (last) rec.desc[1 + tiles] = kTileEnd | (any ? 0u : kTileEmptyItem);
      rec.first = 1;
      rec.end = (int16_t)(1 + tiles + (last ? 1 : 0));
      mbar_arrive(&sm.rec_full[n % kRecords]);
    }
  }
  if (!WAIT(&sm.rec_empty[n % kRecords], ((n / kRecords) & 1) ^ 1, 0)) return;
  sm.rec[n % kRecords].work = -1;
  mbar_arrive(&sm.rec_full[n % kRecords]);
}

static void producer() {
  static unsigned char nothing[1];
  producer_role<C>(sm, prm, nothing, nothing, &tm_q, &tm_k, &tm_v, &tm_kc, &tm_vm);
}

// the waits and arrivals of mma_qk_role, mma_pv_role and softmax_role
template <class F, class G>
static void walk(int warps, F tile, G item_end) {
  Cursor<C> cur;
  for (;;) {
    const uint32_t d = next_desc(sm, cur, wait_limit, nullptr, [&](uint32_t r) {
      for (int i = 0; i < warps; ++i) mbar_arrive(&sm.rec_empty[r]);
    });
    if (d >= kDescNone) return;
    if (!((d & kTileEnd) ? item_end((d & kTileEmptyItem) != 0) : tile((d & kTileFirst) != 0))) return;
  }
}
static void mma_qk() {
  uint32_t g = 0, n_item = 0;
  walk(1, [&](bool first) {
    if (first && !WAIT(&sm.q_full, n_item++ & 1, 0)) return false;
    if (!WAIT(&sm.k_full[g % kKStages], (g / kKStages) & 1, 0)) return false;
    if (g >= 2 && !WAIT(&sm.pv_done[g & 1], ((g - 2) >> 1) & 1, 0)) return false;
    mbar_arrive(&sm.k_empty[g % kKStages]);
    mbar_arrive(&sm.s_full[g & 1]);
    ++g;
    return true;
  }, [&](bool empty) { if (!empty) mbar_arrive(&sm.q_empty); return true; });
}
static void mma_pv() {
  uint32_t g = 0, n_item = 0;
  walk(1, [&](bool first) {
    if (!WAIT(&sm.v_full[g % kVStages], (g / kVStages) & 1, 0)) return false;
    if (first && n_item++ > 0 && !WAIT(&sm.o_free, (n_item - 2) & 1, 0)) return false;
    for (int h = 0; h < 2; ++h)
      if (!WAIT(&sm.p_full[h][g & 1], (g >> 1) & 1, 0)) return false;
    mbar_arrive(&sm.v_empty[g % kVStages]);
    mbar_arrive(&sm.pv_done[g & 1]);
    ++g;
    return true;
  }, [&](bool) { return true; });
}
static void softmax(int h) {
  uint32_t g = 0, n_merge = 0;
  walk(4, [&](bool) {
    if (!WAIT(&sm.s_full[g & 1], (g >> 1) & 1, 0)) return false;
    for (int i = 0; i < 4; ++i) mbar_arrive(&sm.p_full[h][g & 1]);
    ++g;
    return true;
  }, [&](bool empty) {
    if (empty) return true;
    if (!WAIT(&sm.pv_done[(g - 1) & 1], ((g - 1) >> 1) & 1, 0)) return false;
    mbar_arrive(&sm.x_full);
    if (!WAIT(&sm.x_full, n_merge++ & 1, 0)) return false;
    for (int i = 0; i < 4; ++i) mbar_arrive(&sm.o_free);
    return true;
  });
}
static void softmax0() { softmax(0); }
static void softmax1() { softmax(1); }

static void (*const roles[])() = {router, producer, mma_qk, mma_pv, softmax0, softmax1};
static void entry(int i) {
  roles[i]();
  current->done = true;
  yield();
}

static bool run(unsigned seed) {
  memset(&sm, 0, sizeof(sm));
  for (int r = 0; r < kRecords; ++r) { mbar_init(&sm.rec_full[r], 1); mbar_init(&sm.rec_empty[r], kRecReaders); }
  for (int s = 0; s < kKStages; ++s) { mbar_init(&sm.k_full[s], 1); mbar_init(&sm.k_empty[s], 1); }
  for (int s = 0; s < kVStages; ++s) { mbar_init(&sm.v_full[s], 1); mbar_init(&sm.v_empty[s], 1); }
  mbar_init(&sm.q_full, 1); mbar_init(&sm.q_empty, 1); mbar_init(&sm.x_full, 2); mbar_init(&sm.o_free, 8);
  for (int b = 0; b < 2; ++b) {
    mbar_init(&sm.s_full[b], 1); mbar_init(&sm.pv_done[b], 1);
    mbar_init(&sm.p_full[0][b], 4); mbar_init(&sm.p_full[1][b], 4);
  }
  for (auto& l : loads) l.clear();
  stalled = false;
  tasks.clear();
  std::mt19937 rng(seed);
  // every role has a pace of its own, so that any of them may run far ahead of, or behind, the others
  std::vector<unsigned> pace;
  for (int i = 0; i < 6; ++i) {
    auto t = std::make_unique<Task>();
    getcontext(&t->ctx);
    t->ctx.uc_stack.ss_sp = t->stack.data();
    t->ctx.uc_stack.ss_size = t->stack.size();
    t->ctx.uc_link = nullptr;
    makecontext(&t->ctx, (void (*)())entry, 1, i);
    tasks.push_back(std::move(t));
    pace.push_back(1u << (rng() % 12));
  }
  for (;;) {
    std::vector<int> can;
    uint64_t sum = 0;
    bool all_done = true;
    for (int i = 0; i < 6; ++i) {
      const Task& t = *tasks[i];
      all_done &= t.done;
      if (!t.done && (!t.bar || stalled || complete(*t.bar, t.parity))) { can.push_back(i); sum += pace[i]; }
    }
    if (all_done) break;
    if (can.empty()) {
      printf("seed %u: every role waits; K %zu, V %zu tiles loaded\n", seed, loads[1].size(), loads[2].size());
      stalled = true;                            // all waits give up, the roles leave
      continue;
    }
    uint64_t x = rng() % sum;
    int pick = can[0];
    for (int i : can) {
      pick = i;
      if (x < pace[i]) break;
      x -= pace[i];
    }
    current = tasks[pick].get();
    swapcontext(&main_ctx, &current->ctx);
  }
  if (stalled) return false;
  std::vector<std::pair<int, int>> want[3];
  for (size_t w = 0; w < items.size(); ++w) {
    const int at = 100000 * (int)(w % 3) + 1000000 * (int)(w % 2);
    bool any = false;
    for (size_t t = 0; t < items[w].size(); ++t)
      for (int e = 0; e < items[w][t]; ++e) {
        if (!any) want[0].push_back({0, (int)w * 128 + at});
        any = true;
        want[1].push_back({1, (int)(t * 128 + e) * 128 + at});
        want[2].push_back({2, (int)(t * 128 + e) * 128 + at});
      }
  }
  for (int i = 0; i < 3; ++i)
    if (loads[i] != want[i]) {
      printf("seed %u: other loads than the records ask for (side %d)\n", seed, i);
      return false;
    }
  return true;
}

int main(int argc, char** argv) {
  items.push_back({});
  for (int i = 2; i < argc; ++i) {
    if (!strcmp(argv[i], "/")) items.push_back({});
    else items.back().push_back(atoi(argv[i]));
  }
  if (items.back().empty()) items.pop_back();
  const unsigned seeds = (unsigned)atoi(argv[1]);
  for (unsigned s = 0; s < seeds; ++s)
    if (!run(s)) return 1;
  printf("ok\n");
  return 0;
}
