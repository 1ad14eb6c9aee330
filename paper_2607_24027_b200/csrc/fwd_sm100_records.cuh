// The routing records of the kernel with one query block per CTA, how its roles walk them, and the role that loads what
// they ask for.
//
// Included by fwd_sm100.cu behind fwd_sm100_common.cuh and its WAIT / PROF macros, and nothing here needs a GPU to
// run: tests/record_ring.cpp compiles it for the host, with mbarriers and TMA loads of its own, and steps the roles
// through random interleavings.
#pragma once

#include <type_traits>

namespace sol {
namespace fwd {
namespace {

constexpr int kKStages = 2;                      // ring of K tiles
constexpr int kVStages = 2;                      // ring of V tiles (its own ring: the score GEMMs run ahead of P V)
constexpr int kGroup = 32;                       // pooled keys scored per router step (one per lane)
constexpr int kRecords = 4;                      // ring of routing records
constexpr int kRecReaders = 11;                  // the producer, two MMA warps and eight softmax warps hand a record back

// Compile-time shape of one kernel instance.
template <int D, int BLK>
struct Cfg {
  static constexpr int kD = D;                     // head dimension
  static constexpr int kBlk = BLK;                 // block_q = block_k = key columns of a tile
  static constexpr int kHalf = BLK / 2;            // key columns per softmax warpgroup
  static constexpr int kBoxes = D / 64;            // 64-channel TMA boxes per tile row
  static constexpr int kQBytes = kRowsQ * D * 2;   // the query tile
  static constexpr int kTileBytes = BLK * D * 2;   // one K-like or V-like tile
  static constexpr int kQBoxBytes = kRowsQ * 128;  // one box of the query tile (64 channels x 128 rows)
  static constexpr int kBoxBytes = BLK * 128;      // one box of a K-like / V-like tile
  static_assert(D == 64 || D == 128, "head dimension");
  static_assert(BLK == 64 || BLK == 128, "block size");
};

// The router turns every chunk of `block` key blocks into a record: a flat list of tile descriptors
// that the other roles only have to read.  A descriptor is (row coordinate << 5) | flags; the
// coordinate is the first key row of an exact tile or the first pooled row of an approximate one.
constexpr uint32_t kTileApprox = 1;      // approximate-branch tile (pooled keys / mean values)
constexpr uint32_t kTileFirst = 2;       // first tile of its work item: Q_i is loaded, accumulators start afresh
constexpr uint32_t kTileEnd = 4;         // not a tile: the work item ends here
constexpr uint32_t kTileEmptyItem = 8;   // on an end entry: the item had no tile at all
constexpr uint32_t kDescStop = 0xffffffffu, kDescAbort = 0xfffffffeu, kDescNone = 0xfffffffdu;

template <class C>
struct alignas(16) Record {
  float bias[C::kBlk];          // approximate-tile column bias: log2(n_j) / (scale * log2 e), or -inf
  int32_t work;                 // bh * Nq + i, or -1: no more work
  int32_t b, h;                 // batch and head of the work item
  int32_t q_row;                // first query row of the work item
  int16_t first, end;           // descriptors [first, end) are valid (slot 0 is kept for the approximate tile)
  uint32_t desc[C::kBlk + 2];
};

template <class C>
struct Shared {
  float kc_stage[2][kGroup * C::kD];   // router: fp32 pooled keys of the group being scored / the next one
  float qbar_s[C::kD];                 // router: pooled query of the current work item
  Record<C> rec[kRecords];
  float2 ml[2][kRowsQ];         // (m_h, l_h) exchange between the softmax warpgroups
  uint64_t rec_full[kRecords], rec_empty[kRecords];
  uint64_t k_full[kKStages], k_empty[kKStages], v_full[kVStages], v_empty[kVStages];
  uint64_t q_full, q_empty;
  uint64_t s_full[2], p_full[2][2], pv_done[2];   // indexed by score buffer (and warpgroup)
  uint64_t x_full;              // rendezvous of the two softmax warpgroups at the end of a work item
  uint64_t o_free;              // all 8 softmax warps have read both accumulators of the finished work item
  uint64_t kc_full[2];          // router staging buffers filled
  uint64_t mma_drain[2];        // abort path only: all MMAs issued by a role have retired
  uint32_t tmem_base;
  int abort_flag;
};

// ------------------------------------------------------------------------------------------------
// Every consumer role (producer, the two MMA warps, both softmax warpgroups) walks the record
// ring with a cursor of its own and sees the same flat stream of descriptors.
template <class C>
struct Cursor {
  uint32_t n_rec = 0;
  int e = 0, end = 0;
  const Record<C>* rec = nullptr;   // the open record (valid until the next call)
};

// `release` is called when the cursor is done with a record (arrives on rec_empty as appropriate
// for the role).  Returns kDescStop at the end of the stream, kDescAbort when a bounded wait
// expired and, with block = false, kDescNone when the next record has not been written yet.
template <class C, class Release>
__device__ __forceinline__ uint32_t next_desc(Shared<C>& sm, Cursor<C>& c, long long wait_limit, long long* wait_acc,
                                              Release release, bool block = true) {
  for (;;) {
    if (c.e < c.end) return c.rec->desc[c.e++];
    if (c.rec) {
      release(c.n_rec % kRecords);
      c.rec = nullptr;
      ++c.n_rec;
    }
    const uint32_t r = c.n_rec % kRecords;
    if (!block && !mbar_try_wait(&sm.rec_full[r], (c.n_rec / kRecords) & 1)) return kDescNone;
#ifdef SOL_PROFILE
    const long long t = clock64();
#endif
    const bool ok = mbar_wait(&sm.rec_full[r], (c.n_rec / kRecords) & 1, &sm.abort_flag, wait_limit);
#ifdef SOL_PROFILE
    if (wait_acc) *wait_acc += clock64() - t;
#endif
    if (!ok) return kDescAbort;
    if (sm.rec[r].work < 0) return kDescStop;        // stays on this record: every further call stops too
    c.rec = &sm.rec[r];
    c.e = c.rec->first;
    c.end = c.rec->end;
  }
}

// ------------------------------------------------------------------------------------------------
// producer: one thread.  K and V tiles have rings of their own, and the K loads run kLead tiles
// ahead of the V loads: that is the order in which the slots come free (a K slot when its score
// GEMM retires, a V slot a softmax pass and a P V later), so an in-order thread seldom waits for a
// slot while another load could go.  The tiles whose V load is still owed are kept by value and their
// records handed back with the K side: a record kept for an owed tile would also keep the ones behind it
// that hold no tile (keep-or-drop mode), which the router may have to write again before the K side can go on.
template <class C>
__device__ void producer_role(Shared<C>& sm, const Params& p, unsigned char* sQ, unsigned char* sKV,
                              const CUtensorMap* tm_q, const CUtensorMap* tm_k, const CUtensorMap* tm_v,
                              const CUtensorMap* tm_kc, const CUtensorMap* tm_vm) {
  constexpr int kLead = 2;                           // owed0 and owed1 below
  constexpr int kTileBytes = C::kTileBytes;
  const long long wait_limit = p.wait_limit;
  uint32_t n_k = 0, n_v = 0, n_item = 0;
  Cursor<C> cur;
  struct Tile { uint32_t dsc; int b, h; } owed0{}, owed1{};    // oldest first
  PROF_DECL
  // pooled = true: KC / mean-V operands, dense [B*H][Nk][d]; else q, k, v in the caller's layout.
  // A tile is C::kBoxes boxes of 64 channels, each kBox bytes long in shared memory.
  auto load_tile = [&](auto bytes_c, auto box_c, const CUtensorMap* tm, uint64_t* full, unsigned char* dst, int row,
                       int b, int h, bool pooled) {
    constexpr int kBytes = decltype(bytes_c)::value, kBox = decltype(box_c)::value;
    mbar_arrive_expect_tx(full, kBytes);
    const bool rows_inner = pooled || p.rows_inner;
    const int c1 = rows_inner ? row : h, c2 = rows_inner ? h : row;
    tma_load_4d(dst, tm, full, 0, c1, c2, b);
    if constexpr (C::kBoxes == 2) tma_load_4d(dst + kBox, tm, full, 64, c1, c2, b);
  };
  using QBytes = std::integral_constant<int, C::kQBytes>;
  using QBox = std::integral_constant<int, C::kQBoxBytes>;
  using TBytes = std::integral_constant<int, C::kTileBytes>;
  using TBox = std::integral_constant<int, C::kBoxBytes>;
  auto release = [&](uint32_t r) { mbar_arrive(&sm.rec_empty[r]); };
  bool k_end = false, have_k = false, ok = true;
  uint32_t dk = 0;
  for (;;) {
    // K side (and Q): up to kLead tiles ahead of the V side
    while (!k_end && (int)(n_k - n_v) < kLead) {
      if (!have_k) {
        // (never sleep on the router while a V load is owed: the router may itself wait for what that load sets going)
        dk = next_desc(sm, cur, wait_limit, PROF_ACC(0), release, n_k == n_v);        // prof 0: no record yet
        if (dk == kDescNone) break;
        if (dk == kDescAbort) { ok = false; break; }
        if (dk == kDescStop) { k_end = true; break; }
        have_k = true;
      }
      if (dk & kTileEnd) { have_k = false; continue; }
      if (dk & kTileFirst) {
        // Q_i for this work item.  The slot frees when the previous item's last score GEMM
        // retires; until then serve the V side.
        const uint32_t par = (n_item & 1) ^ 1;
        if (n_k != n_v && !mbar_try_wait(&sm.q_empty, par)) break;
        if (!WAIT(&sm.q_empty, par, 2)) { ok = false; break; }                  // prof 2: Q slot busy
        load_tile(QBytes{}, QBox{}, tm_q, &sm.q_full, sQ, cur.rec->q_row, cur.rec->b, cur.rec->h, false);
        ++n_item;
        dk &= ~kTileFirst;
      }
      have_k = false;
      const uint32_t s = n_k % kKStages;
      if (!WAIT(&sm.k_empty[s], ((n_k / kKStages) & 1) ^ 1, 1)) { ok = false; break; }   // prof 1: K ring full
      const Tile t{dk, cur.rec->b, cur.rec->h};
      {
        PROF_T0
        load_tile(TBytes{}, TBox{}, (dk & kTileApprox) ? tm_kc : tm_k, &sm.k_full[s], sKV + (size_t)s * kTileBytes,
                  (int)(dk >> 5), t.b, t.h, (dk & kTileApprox) != 0);
        PROF_ADD(4)                                                                    // prof 4: issuing K copies
      }
      if (n_k == n_v) owed0 = t;
      else owed1 = t;
      ++n_k;
    }
    if (!ok) break;
    if (n_k == n_v) {
      if (k_end) break;
      continue;
    }
    // V side: the oldest tile whose K is already on its way
    const Tile t = owed0;
    owed0 = owed1;
    const uint32_t s = n_v % kVStages;
    if (!WAIT(&sm.v_empty[s], ((n_v / kVStages) & 1) ^ 1, 3)) { ok = false; break; }     // prof 3: V ring full
    {
      PROF_T0
      load_tile(TBytes{}, TBox{}, (t.dsc & kTileApprox) ? tm_vm : tm_v, &sm.v_full[s],
                sKV + (size_t)(kKStages + s) * kTileBytes, (int)(t.dsc >> 5), t.b, t.h, (t.dsc & kTileApprox) != 0);
      PROF_ADD(5)                                                                      // prof 5: issuing V copies
    }
    ++n_v;
  }
  if (!ok) flag_abort(sm, p, 200);
  PROF_FLUSH(1);
  if (sm.abort_flag) {
    // let copies that are still in flight land before the CTA's shared memory goes away
    int never = 0;                                   // this drain must not be cut short by the abort flag
    if (n_item > 0) mbar_wait(&sm.q_full, (n_item - 1) & 1, &never, wait_limit);
    for (uint32_t back = 0; back < kKStages && back < n_k; ++back) {
      const uint32_t n = n_k - 1 - back;
      mbar_wait(&sm.k_full[n % kKStages], (n / kKStages) & 1, &never, wait_limit);
    }
    for (uint32_t back = 0; back < kVStages && back < n_v; ++back) {
      const uint32_t n = n_v - 1 - back;
      mbar_wait(&sm.v_full[n % kVStages], (n / kVStages) & 1, &never, wait_limit);
    }
  }
}

}  // namespace
}  // namespace fwd
}  // namespace sol
