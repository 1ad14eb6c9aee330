// Sol-Attn fused forward (Algorithm 1) for sm_100a: TMA + tcgen05.mma + TMEM.
//
// Persistent kernel, one CTA of 384 threads per SM, compiled for d in {64, 128} and blocks of 128 or 64 tokens (64: for
// calls of at most one query block per SM; fwd_sm100_b64.cu takes the others).  A CTA owns one query block at a time and is
// split into warp roles that talk through mbarriers:
//
//   router   (warp 8)  pulls (head, query block) work items from a global counter and walks the
//                      pooled keys in chunks of `block` blocks.  For every block it evaluates the
//                      proxy s_ij = scale * Qbar_i . KC_j (Eq. 3) in fp32 and compares it with
//                      tau_i (Eq. 4).  The decision only ever lives in a small shared-memory
//                      record (flat list of tile descriptors + per-column bias); nothing of the
//                      proxy map goes to global memory.
//   producer (warp 9, one lane) reads the records and issues TMA loads: one approximate tile per
//                      chunk (KC chunk, mean-V chunk) and K_j / V_j ONLY for routed blocks.
//   mma      (warps 10, 11) issue tcgen05.mma: warp 10 the score GEMMs S = Q K^T, warp 11 the value
//                      GEMMs O += P V; each warp runs in lockstep and one elected lane issues.  S
//                      goes to one of two TMEM score buffers, so the scores of tile g+1 are
//                      computed while tile g is in softmax.
//   softmax  (warps 0-3 and 4-7) two warpgroups; thread = query row; group h owns key columns
//                      [block/2 * h, block/2 * (h+1)) of EVERY tile and keeps its own running
//                      (m_h, l_h) and its own accumulator O_h in TMEM; the two partial results are
//                      merged when the query block is finished.  Both branches of the method
//                      update the same state: an approximate tile is an ordinary tile whose
//                      columns carry the bias log2(n_j) (Eqs. 9-10: multiplicity n_j in the
//                      denominator, mean value times n_j in the numerator) or -inf for routed /
//                      padded columns.  O_h is rescaled lazily, only when the running maximum
//                      grows by more than 2^8.
//
// The query tile of the MMAs always has 128 rows (the M of a one-CTA tcgen05.mma at full rate); with 64-token
// blocks its upper 64 rows belong to the next query block, take part in the arithmetic and are never stored.
//
// TMEM (512 columns): S0 [0, block)  S1 [block, 2 block)  O0 [256, 256 + d)  O1 [256 + d, 256 + 2 d);
// P_h (bf16) of a tile overwrites the start of group h's half of that tile's S buffer.
//
// Every mbarrier wait is bounded: when one expires the CTA records SOL_ERR_DEVICE_TIMEOUT in the
// workspace status word, all roles drain, TMEM is released and the kernel returns.
#include "fwd_sm100_common.cuh"

// Every role has `sm` and `wait_limit` in scope; WAIT is a bounded wait on one of its barriers.
#if defined(SOL_PROFILE) || defined(SOL_ITEMTRACE)
#include "fwd_sm100_prof.cuh"
#endif
#ifdef SOL_PROFILE
#define WAIT(bar, parity, slot) SOL_WAIT(bar, parity, slot)
#else
#define WAIT(bar, parity, slot) mbar_wait((bar), (parity), &sm.abort_flag, wait_limit)
#define PROF_DECL
#define PROF_COUNT(slot)
#define PROF_FLUSH(role)
#define PROF_ACC(slot) nullptr
#define PROF_T0
#define PROF_ADD(slot)
#endif
#ifndef SOL_ITEMTRACE
#define ITRACE(item, slot)
#define ITRACE_VAL(item, slot, val)
#define CTATRACE(slot, val)
#endif
#include "fwd_sm100_records.cuh"

namespace sol {
namespace fwd {
namespace {

constexpr int kWarpQK = 10;                      // warp 11 issues P V
constexpr int kTmemS = 0, kTmemO = 256;

// ------------------------------------------------------------------------------------------------
// router: one warp
// kFromMask: the decisions were taken by the routing pre-pass and are read back from the mask (one bit per
// (query block, key block)) instead of being scored here.
template <class C, bool kFromMask>
__device__ void router_role(Shared<C>& sm, const Params& p, int lane) {
  constexpr int kD = C::kD, kBlk = C::kBlk, kPieces = C::kD / 4;   // 16-byte pieces per pooled key
  const unsigned full = 0xffffffffu;
  const long long wait_limit = p.wait_limit;
  uint32_t n_rec = 0, n_copy = 0, n_use = 0;   // records written; staging copies issued / consumed
  uint32_t n_item = 0;
  const int n_chunks = ceil_div(p.Nk, kBlk);
  const int mask_words = ceil_div(p.Nk, 32);
  const float inv_sl2 = 1.f / (p.scale * 1.4426950408889634f);   // biases are stored in raw-score units
  constexpr bool from_mask = kFromMask;
  const float bias_full = log2f((float)kBlk) * inv_sl2;                          // log2 n_j of a full block ...
  const float bias_last = log2f((float)(p.N - (p.Nk - 1) * kBlk)) * inv_sl2;     // ... and of the ragged last one
  bool alive = true;
  PROF_DECL
  if (lane == 0) CTATRACE(0, prof::gtimer());
  while (alive) {
    int w = 0;
    if (lane == 0) w = atomicAdd(p.status + kStatusTileCounter, 1);
    w = __shfl_sync(full, w, 0);
    if (w >= p.total_work) break;
    if (lane == 0) ITRACE(n_item, 0);
    const int bh = w / p.Nq, i = w - bh * p.Nq;
    // the pooled query of this work item goes to shared memory (one 16-byte piece per lane)
    float tau_i = 0.f;
    if (p.mode != SOL_MODE_DENSE && !from_mask) {
      __syncwarp();
      if (lane < kPieces)
        reinterpret_cast<float4*>(sm.qbar_s)[lane] =
            __ldg(reinterpret_cast<const float4*>(p.qbar + ((size_t)bh * p.Nq + i) * kD) + lane);
      tau_i = p.tau[(size_t)bh * p.Nq + i];
      __syncwarp();
    }
    const float* kc_head = p.kc + (size_t)bh * p.Nk * kD;
    int count = 0;
    bool item_has_tiles = false;
    // Bulk-copy one group of 32 pooled keys (contiguous in memory) into a staging buffer;
    // the copy of group n+1 is in flight while group n is scored.
    auto stage_group = [&](int jb) {
      if (p.mode == SOL_MODE_DENSE || from_mask || jb >= p.Nk) return;
      __syncwarp();                                  // every lane is done reading this buffer
      if (lane == 0) {
        const uint32_t buf = n_copy & 1;
        const uint32_t bytes = (uint32_t)min(kGroup, p.Nk - jb) * kD * 4;
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&sm.kc_full[buf], bytes);
        bulk_load_1d(sm.kc_stage[buf], kc_head + (size_t)jb * kD, bytes, &sm.kc_full[buf]);
      }
      ++n_copy;
    };
    stage_group(0);
    for (int t = 0; t < n_chunks; ++t) {
      Record<C>& rec = sm.rec[n_rec % kRecords];
      if (!WAIT(&sm.rec_empty[n_rec % kRecords], ((n_rec / kRecords) & 1) ^ 1, 0)) {   // prof 0: record ring full
        if (lane == 0) flag_abort(sm, p, 100);
        alive = false;
        break;
      }
      const int j0 = t * kBlk;
      int n_sel = 0;
      bool any_unselected = false;
#pragma unroll 1
      for (int g = 0; g < kBlk / 32; ++g) {
        const int jbase = j0 + g * 32;
        bool sel;
        const int j = jbase + lane;
        if (p.mode == SOL_MODE_DENSE) {
          sel = j < p.Nk;
        } else if (from_mask) {
          sel = (j < p.Nk) && ((p.mask_out[(size_t)w * mask_words + jbase / 32] >> lane) & 1u);
        } else {
          // lane l scores pooled key jbase + l against the staged rows.  Lane l starts at 16-byte
          // piece l of its row and of the query and walks round, so that the lanes spread over the
          // shared-memory bank groups although the rows are a multiple of 128 bytes apart.
          float dot = 0.f;
          if (jbase < p.Nk) {
            const uint32_t buf = n_use & 1;
            if (!WAIT(&sm.kc_full[buf], (n_use >> 1) & 1, 1)) {                         // prof 1: pooled keys not staged
              if (lane == 0) flag_abort(sm, p, 102);
              alive = false;
              break;
            }
            ++n_use;
            stage_group(jbase + kGroup);              // next group of this work item, if any
            const float4* row = reinterpret_cast<const float4*>(sm.kc_stage[buf] + lane * kD);
            const float4* qv = reinterpret_cast<const float4*>(sm.qbar_s);
            float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
            for (int c = 0; c < kPieces; ++c) {
              const int piece = (c + lane) & (kPieces - 1);
              const float4 kk = row[piece];
              const float4 qq = qv[piece];
              a0 = fmaf(qq.x, kk.x, a0);
              a1 = fmaf(qq.y, kk.y, a1);
              a2 = fmaf(qq.z, kk.z, a2);
              a3 = fmaf(qq.w, kk.w, a3);
            }
            dot = (a0 + a1) + (a2 + a3);
          }
          sel = (j < p.Nk) && (p.scale * dot > tau_i);
          if (p.forced && j < p.Nk && p.forced[j]) sel = true;
        }
        const unsigned m = __ballot_sync(full, sel);
        const bool valid = j < p.Nk;
        any_unselected |= (valid && !sel);
        rec.bias[g * 32 + lane] = (valid && !sel) ? (j == p.Nk - 1 ? bias_last : bias_full) : -INFINITY;
        if (sel) rec.desc[1 + n_sel + __popc(m & ((1u << lane) - 1u))] = (uint32_t)(j * kBlk) << 5;
        n_sel += __popc(m);
        if (p.mask_out && !from_mask && lane == 0 && jbase < p.Nk) p.mask_out[(size_t)w * mask_words + jbase / 32] = m;
      }
      if (!alive) break;
      any_unselected = __any_sync(full, any_unselected);
      count += n_sel;
      const bool has_approx = p.mode == SOL_MODE_SOL && any_unselected;
      const int first = has_approx ? 0 : 1;
      int end = 1 + n_sel;                   // n_sel <= block
      __syncwarp();
      if (lane == 0) {
        rec.work = w;
        rec.b = bh / p.st.H;
        rec.h = bh - rec.b * p.st.H;
        rec.q_row = i * kBlk;
        if (has_approx) rec.desc[0] = ((uint32_t)j0 << 5) | kTileApprox;
        if (!item_has_tiles && end > first) rec.desc[first] |= kTileFirst;
        if (t == n_chunks - 1) rec.desc[end] = kTileEnd | ((item_has_tiles || end > first) ? 0u : kTileEmptyItem);
        rec.first = (int16_t)first;
        rec.end = (int16_t)(end + (t == n_chunks - 1 ? 1 : 0));
      }
      item_has_tiles |= end > first;
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.rec_full[n_rec % kRecords]);
      if (lane == 0 && t == 0) ITRACE(n_item, 1);
      if (lane == 0 && t == n_chunks - 1) ITRACE(n_item, 2);
      ++n_rec;
    }
    if (alive && lane == 0 && p.counts) p.counts[w] = count;
    ++n_item;
  }
  if (lane == 0) { CTATRACE(1, prof::gtimer()); CTATRACE(2, (long long)n_item); }
  PROF_FLUSH(0);
  if (!alive) {
    // let a staging copy that is still in flight land before the CTA's shared memory goes away
    int never = 0;                                   // this drain must not be cut short by the abort flag
    for (; n_use != n_copy; ++n_use) mbar_wait(&sm.kc_full[n_use & 1], (n_use >> 1) & 1, &never, wait_limit);
  }
  // end-of-stream record
  if (alive) {
    if (mbar_wait(&sm.rec_empty[n_rec % kRecords], ((n_rec / kRecords) & 1) ^ 1, &sm.abort_flag, wait_limit)) {
      if (lane == 0) {
        sm.rec[n_rec % kRecords].work = -1;
        mbar_arrive(&sm.rec_full[n_rec % kRecords]);
      }
    } else if (lane == 0) {
      flag_abort(sm, p, 101);
    }
  }
}

// ------------------------------------------------------------------------------------------------
// MMA issue is split over two single-thread roles so that neither the waits nor the scalar
// bookkeeping of one kind of MMA delays the other; the tensor pipe arbitrates between them and all
// ordering is carried by the mbarriers.
//
// Abort path of an MMA-issuing role: TMEM must not be released while MMAs are still writing to it, so
// the role asks for a completion signal behind everything it has issued and waits for it (bounded).
template <class C>
__device__ __forceinline__ void drain_mmas(Shared<C>& sm, uint64_t* bar, bool leader, long long wait_limit) {
  if (leader) mma_commit(bar);
  int never = 0;
  mbar_wait(bar, 0, &never, wait_limit);
}

// S_b = Q K^T (warp 10)
template <class C>
__device__ void mma_qk_role(Shared<C>& sm, const Params& p, unsigned char* sQ, unsigned char* sKV, uint32_t tmem) {
  constexpr int kD = C::kD, kBlk = C::kBlk, kTileBytes = C::kTileBytes;
  const long long wait_limit = p.wait_limit;
  const uint32_t idesc_qk = make_idesc_bf16(kRowsQ, kBlk, false, false);
  const uint32_t q_lo = (smem_addr(sQ) >> 4) | (1u << 16);
  const uint32_t kv_lo = (smem_addr(sKV) >> 4) | (1u << 16);
  uint32_t n_item = 0, g = 0;
  uint32_t slot = 0, slot_parity = 0;          // ring position of K(g)
  Cursor<C> cur;
  PROF_DECL
  // The whole warp runs this role in lockstep and one elected lane issues: with warp-uniform control
  // flow and operands the compiler keeps descriptors and addresses in uniform registers, where the
  // MMA instruction wants them, instead of moving them over from a single divergent lane's registers.
  const bool leader = elect_one();
  auto release = [&](uint32_t r) { if (leader) mbar_arrive(&sm.rec_empty[r]); };
  bool ok = true;
  for (;;) {
    const uint32_t dsc = next_desc(sm, cur, wait_limit, PROF_ACC(0), release);        // prof 0: no record yet
    if (dsc == kDescAbort) { ok = false; break; }
    if (dsc == kDescStop) break;
    if (dsc & kTileEnd) {                         // every MMA that reads Q_i has been issued
      if (!(dsc & kTileEmptyItem) && leader) mma_commit(&sm.q_empty);
      continue;
    }
    const bool it_first = (dsc & kTileFirst) != 0;
    if (it_first) {
      if (leader) ITRACE(n_item, 3);
      if (!WAIT(&sm.q_full, n_item & 1, 1)) { ok = false; break; }                    // prof 1: Q not loaded
      ++n_item;
    }
    const uint32_t b = g & 1;
    if (!WAIT(&sm.k_full[slot], slot_parity, 2)) { ok = false; break; }               // prof 2: K not loaded
    if (g >= 2) {
      // P overwrites S: the P V of tile g-2 must have read P out of this buffer
      if (!WAIT(&sm.pv_done[b], ((g - 2) >> 1) & 1, 3)) { ok = false; break; }        // prof 3: score buffer busy
    }
    tc_fence_after();
    {
      PROF_T0
      const uint32_t k_lo = kv_lo + slot * (kTileBytes >> 4);
      const uint32_t d_tmem = tmem + kTmemS + b * kBlk;
#pragma unroll
      for (int ks = 0; ks < kD / 16; ++ks) {
        // K-step ks: 16 channels = 32 bytes inside box ks / 4
        const uint32_t off_q = ((ks / 4) * C::kQBoxBytes + (ks % 4) * 32) >> 4;
        const uint32_t off_k = ((ks / 4) * C::kBoxBytes + (ks % 4) * 32) >> 4;
        const uint64_t da = desc_from_lo(q_lo + off_q), db = desc_from_lo(k_lo + off_k);
        if (leader) mma_ss(d_tmem, da, db, idesc_qk, ks > 0);
      }
      if (leader) {
        mma_commit(&sm.k_empty[slot]);
        mma_commit(&sm.s_full[b]);
      }
      PROF_ADD(6)                                                                      // prof 6: issuing Q K^T
      if (it_first && leader) ITRACE(n_item - 1, 4);
    }
    ++g;
    if (++slot == kKStages) { slot = 0; slot_parity ^= 1; }
  }
  if (!ok && leader) flag_abort(sm, p, 300);
  __syncwarp();
  if (sm.abort_flag) drain_mmas(sm, &sm.mma_drain[0], leader, wait_limit);
  if (leader) PROF_FLUSH(2);
}

// O_h (+)= P_h V[half h of the tile's keys], h = 0, 1 (warp 11)
template <class C>
__device__ void mma_pv_role(Shared<C>& sm, const Params& p, unsigned char* sKV, uint32_t tmem) {
  constexpr int kD = C::kD, kBlk = C::kBlk, kHalf = C::kHalf, kTileBytes = C::kTileBytes;
  const long long wait_limit = p.wait_limit;
  const uint32_t idesc_pv = make_idesc_bf16(kRowsQ, kD, false, true);
  // V is the MN-major operand: its 64-channel boxes are C::kBoxBytes apart (leading offset), groups of
  // 8 key rows 1024 bytes apart; a K-step of 16 keys advances the start by 2048 bytes.
  const uint32_t kv_lo = (smem_addr(sKV + kKStages * kTileBytes) >> 4) | ((uint32_t)(C::kBoxBytes >> 4) << 16);
  uint32_t g = 0, n_item = 0;
  uint32_t slot = 0, slot_parity = 0;          // ring position of V(g)
  Cursor<C> cur;
  const bool leader = elect_one();             // warp-uniform role, one issuing lane (see mma_qk_role)
  auto release = [&](uint32_t r) { if (leader) mbar_arrive(&sm.rec_empty[r]); };
  bool ok = true;
  for (;;) {
    const uint32_t dsc = next_desc(sm, cur, wait_limit, nullptr, release);
    if (dsc == kDescAbort) { ok = false; break; }
    if (dsc == kDescStop) break;
    if (dsc & kTileEnd) continue;
    const uint32_t b = g & 1;
    if (!mbar_wait(&sm.v_full[slot], slot_parity, &sm.abort_flag, wait_limit)) { ok = false; break; }
    const uint32_t v_lo = kv_lo + slot * (kTileBytes >> 4);
    const uint32_t acc_first = (dsc & kTileFirst) ? 0u : 1u;
    if ((dsc & kTileFirst) && n_item++ > 0) {
      // the first P V of a work item overwrites O0 / O1: the previous item's merge must have read them
      if (!mbar_wait(&sm.o_free, (n_item - 2) & 1, &sm.abort_flag, wait_limit)) { ok = false; break; }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (!mbar_wait(&sm.p_full[h][b], (g >> 1) & 1, &sm.abort_flag, wait_limit)) { ok = false; break; }
      tc_fence_after();
#pragma unroll
      for (int ks = 0; ks < kHalf / 16; ++ks) {
        const uint32_t d_o = tmem + kTmemO + h * kD;
        const uint32_t a_p = tmem + kTmemS + b * kBlk + h * kHalf + ks * 8;
        const uint32_t acc = ks > 0 ? 1u : acc_first;
        const uint64_t dv = desc_from_lo(v_lo + ((h * (kHalf * 128) + ks * 2048) >> 4));
        if (leader) mma_ts(d_o, a_p, dv, idesc_pv, acc);
      }
    }
    if (!ok) break;
    if (leader) {
      mma_commit(&sm.v_empty[slot]);
      // (test hook: a withheld completion signal makes the bounded waits on it run out)
      if ((int)g != p.withhold_tile) mma_commit(&sm.pv_done[b]);
    }
    ++g;
    if (++slot == kVStages) { slot = 0; slot_parity ^= 1; }
  }
  if (!ok && leader) flag_abort(sm, p, 301);
  __syncwarp();
  if (sm.abort_flag) drain_mmas(sm, &sm.mma_drain[1], leader, wait_limit);
}

// ------------------------------------------------------------------------------------------------
// softmax + correction + epilogue: two warpgroups of 128 threads; thread = query row, warpgroup h
// owns key columns [kHalf h, kHalf (h+1)) of every tile.
template <class C>
__device__ void softmax_role(Shared<C>& sm, const Params& p, uint32_t tmem, int h, int warp_in_group, int lane) {
  constexpr int kD = C::kD, kBlk = C::kBlk, kHalf = C::kHalf;
  constexpr int kOutCh = kD / 2;                             // output channels written by one warpgroup
  const unsigned full = 0xffffffffu;
  const long long wait_limit = p.wait_limit;
  const uint32_t lane_base = tmem + ((uint32_t)(warp_in_group * 32) << 16);
  const uint32_t t_o = lane_base + kTmemO + h * kD;          // this group's accumulator
  const uint32_t t_o_other = lane_base + kTmemO + (1 - h) * kD;
  const int row = warp_in_group * 32 + lane;
  const float sl2 = p.scale * 1.4426950408889634f;
  uint32_t g = 0, n_merge = 0;
  uint32_t n_item = 0, g_item0 = 0;        // item trace only
  float m_used = -INFINITY, l = 0.f;
  Cursor<C> cur;
  PROF_DECL
  auto release = [&](uint32_t r) {
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm.rec_empty[r]);
  };
  // A wait that gives up must give up for the whole warp: the loop holds warp-synchronising
  // operations (TMEM loads and stores, votes), so the lanes leave together or not at all.
#define SWAIT(bar, parity, slot) __all_sync(full, WAIT(bar, parity, slot))
  // The next descriptor of the open record is read from shared memory while the current tile is being
  // worked on, so that the read's latency is off the path from one tile to the next.
  bool peeked = false;
  uint32_t dsc_peek = 0;
  for (;;) {
    uint32_t dsc;
    if (peeked) {
      dsc = dsc_peek;
      ++cur.e;
    } else {
      dsc = next_desc(sm, cur, wait_limit, PROF_ACC(0), release);                     // prof 0: no record yet
      if (dsc == kDescAbort) { flag_abort(sm, p, 400); break; }
      if (dsc == kDescStop) break;
    }
    peeked = cur.e < cur.end;
    if (peeked) dsc_peek = cur.rec->desc[cur.e];
    const bool first = (dsc & kTileFirst) != 0;

    if (!(dsc & kTileEnd)) {
      const uint32_t b = g & 1;
      const uint32_t t_s = lane_base + kTmemS + b * kBlk + h * kHalf;
      const bool approx = (dsc & kTileApprox) != 0;
      const int cols_valid = approx ? kBlk : min(kBlk, p.N - (int)(dsc >> 5));
      const bool general = approx || cols_valid < kBlk;
      // (no vote on this wait, the one wait of every tile: the 32 lanes poll the same barrier, abort flag
      //  and clock in lockstep and leave the loop together; the rarer waits below are made uniform by a vote)
      if (!WAIT(&sm.s_full[b], (g >> 1) & 1, 1)) { flag_abort(sm, p, 401); break; }   // prof 1: S not ready
      tc_fence_after();
      if (first && warp_in_group == 0 && lane == 0) { ITRACE(n_item, h ? 11 : 5); g_item0 = g; }
      // ---- this group's half row of S (kHalf fp32) into registers with one wait
      uint32_t sr[kHalf];
      PROF_T0
      tmem_ld_cols<kHalf>(t_s, sr);
      tmem_ld_wait();
      PROF_ADD(7)                                                                      // prof 7: loading S
      if (general) {
        // bring the rare tiles (approximate chunk, ragged last block) to the common form
        // logit = sl2 * x by folding the column bias into x; -inf marks masked columns
        if (approx) {
          const float4* bias4 = reinterpret_cast<const float4*>(&cur.rec->bias[h * kHalf]);
#pragma unroll
          for (int c = 0; c < kHalf / 4; ++c) {
            const float4 bb = bias4[c];
            sr[4 * c] = __float_as_uint(__uint_as_float(sr[4 * c]) + bb.x);
            sr[4 * c + 1] = __float_as_uint(__uint_as_float(sr[4 * c + 1]) + bb.y);
            sr[4 * c + 2] = __float_as_uint(__uint_as_float(sr[4 * c + 2]) + bb.z);
            sr[4 * c + 3] = __float_as_uint(__uint_as_float(sr[4 * c + 3]) + bb.w);
          }
        } else {
#pragma unroll
          for (int c = 0; c < kHalf; ++c)
            if (h * kHalf + c >= cols_valid) sr[c] = __float_as_uint(-INFINITY);
        }
      }
      float mx;
      {
        constexpr int kQ = kHalf / 4;
        float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
        for (int c = 0; c < kQ; ++c) {
          m0 = fmaxf(m0, __uint_as_float(sr[c]));
          m1 = fmaxf(m1, __uint_as_float(sr[kQ + c]));
          m2 = fmaxf(m2, __uint_as_float(sr[2 * kQ + c]));
          m3 = fmaxf(m3, __uint_as_float(sr[3 * kQ + c]));
        }
        mx = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3)) * sl2;       // -inf when the whole half is masked
      }
      // ---- running maximum, lazy rescale of O_h
      if (first) {
        m_used = mx;
        l = 0.f;
      } else if (__any_sync(full, mx > m_used + kRescaleThreshold)) {
        const float m_new = fmaxf(m_used, mx);
        const float f = (m_new == -INFINITY) ? 1.f : ex2(m_used - m_new);
        PROF_COUNT(4);                                                                  // prof 4: number of rescales
        // P V of the previous tile must have landed in O_h
        if (!SWAIT(&sm.pv_done[b ^ 1], ((g - 1) >> 1) & 1, 2)) { flag_abort(sm, p, 402); break; }
        tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < kD / 32; ++c) {
          uint32_t o[32];
          tmem_ld_32x32b_x32(t_o + c * 32, o);
          tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 32; ++x) o[x] = __float_as_uint(__uint_as_float(o[x]) * f);
          tmem_st_32x32b_x32(t_o + c * 32, o);
        }
        l *= f;
        m_used = m_new;
      }
      // ---- P = exp2(sl2 * S - m) (scaling and row sum as packed fp32 pairs); P (bf16) back to
      //      TMEM over the start of the half
      {
        const float nm = (m_used == -INFINITY) ? 0.f : -m_used;   // a half that has seen nothing yet: all P = 0
        const float2 sl2_2 = make_float2(sl2, sl2), nm2 = make_float2(nm, nm);
        float2 s_a = make_float2(0.f, 0.f), s_b = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < kHalf; c += 4) {
          const float2 xa = __ffma2_rn(make_float2(__uint_as_float(sr[c]), __uint_as_float(sr[c + 1])), sl2_2, nm2);
          const float2 xb = __ffma2_rn(make_float2(__uint_as_float(sr[c + 2]), __uint_as_float(sr[c + 3])), sl2_2, nm2);
          const float2 ea = make_float2(ex2(xa.x), ex2(xa.y));
          const float2 eb = make_float2(ex2(xb.x), ex2(xb.y));
          s_a = __fadd2_rn(s_a, ea);
          s_b = __fadd2_rn(s_b, eb);
          __nv_bfloat162 lo = __floats2bfloat162_rn(ea.x, ea.y);
          __nv_bfloat162 hi = __floats2bfloat162_rn(eb.x, eb.y);
          sr[c / 2] = *reinterpret_cast<uint32_t*>(&lo);
          sr[c / 2 + 1] = *reinterpret_cast<uint32_t*>(&hi);
        }
        {
          const float2 t = __fadd2_rn(s_a, s_b);
          l += t.x + t.y;
        }
        if constexpr (kHalf == 64) tmem_st_32x32b_x32(t_s, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
        else tmem_st_32x32b_x16(t_s, *reinterpret_cast<uint32_t(*)[16]>(&sr[0]));
      }
      PROF_ADD(8)                                                                      // prof 8: load + arithmetic
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();                                  // one arrival per warp: 4 instead of 128 on the barrier
      if (lane == 0) mbar_arrive(&sm.p_full[h][b]);
      PROF_ADD(9)                                                                      // prof 9: whole tile
#ifdef SOL_PROFILE
      if (approx) { prof.v[10] += clock64() - prof_t0; ++prof.v[0]; }                  // prof 10 / 0: approximate tiles: cycles / count
#endif
      PROF_COUNT(5);                                                                    // prof 5: tiles
      ++g;
      continue;
    }

    // ---- end of the work item: merge the two partial results, O_i = (w0 O0 + w1 O1) / (w0 l0 + w1 l1)
    const int q_row = cur.rec->q_row;
    const int q_rows = min(kBlk, p.N - q_row);
    __nv_bfloat16* orow = p.out + (size_t)cur.rec->b * (size_t)p.st.batch + (size_t)cur.rec->h * (size_t)p.st.head +
                          (size_t)(q_row + row) * (size_t)p.st.row + h * kOutCh;
    PROF_T0
    if (warp_in_group == 0 && lane == 0) {
      ITRACE(n_item, h ? 12 : 6);
      if (h == 0) ITRACE_VAL(n_item, 10, (long long)(g - g_item0));
    }
    if (!(dsc & kTileEmptyItem)) {
      // the last P V of the item (one commit covers both halves)
      if (!SWAIT(&sm.pv_done[(g - 1) & 1], ((g - 1) >> 1) & 1, 3)) { flag_abort(sm, p, 403); break; }   // prof 3
      tc_fence_after();
      if (h == 0 && warp_in_group == 0 && lane == 0) ITRACE(n_item, 7);
      sm.ml[h][row] = make_float2(m_used, l);
      mbar_arrive(&sm.x_full);
      if (!SWAIT(&sm.x_full, n_merge & 1, 6)) { flag_abort(sm, p, 404); break; }      // prof 6: other group not done
      if (warp_in_group == 0 && lane == 0) ITRACE(n_item, h ? 13 : 8);
      const float2 other = sm.ml[1 - h][row];
      const float m = fmaxf(m_used, other.x);
      const float w_own = (m_used == -INFINITY) ? 0.f : ex2(m_used - m);
      const float w_other = (other.x == -INFINITY) ? 0.f : ex2(other.x - m);
      const float inv = 1.f / (l * w_own + other.y * w_other);
      const float c_own = w_own * inv, c_other = w_other * inv;
      // this thread writes channels [kOutCh h, kOutCh (h+1)) of its row
#pragma unroll 1
      for (int c = 0; c < kOutCh / 32; ++c) {
        uint32_t a[32], bb[32];
        tmem_ld_32x32b_x32(t_o + h * kOutCh + c * 32, a);
        tmem_ld_32x32b_x32(t_o_other + h * kOutCh + c * 32, bb);
        tmem_ld_wait();
        if (c == kOutCh / 32 - 1) {
          // both accumulators are in registers: the next item's first P V may overwrite them
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sm.o_free);
        }
        if (row < q_rows) {
#pragma unroll
          for (int x = 0; x < 2; ++x) {                 // 32 bytes (16 channels) per store
            uint32_t pw[8];
#pragma unroll
            for (int y = 0; y < 8; ++y) {
              const int e0 = x * 16 + 2 * y;
              // a partial accumulator that never received a tile may hold anything: weight 0 must win
              const float v0 = (w_own > 0.f ? __uint_as_float(a[e0]) * c_own : 0.f) +
                               (w_other > 0.f ? __uint_as_float(bb[e0]) * c_other : 0.f);
              const float v1 = (w_own > 0.f ? __uint_as_float(a[e0 + 1]) * c_own : 0.f) +
                               (w_other > 0.f ? __uint_as_float(bb[e0 + 1]) * c_other : 0.f);
              __nv_bfloat162 hh = __floats2bfloat162_rn(v0, v1);
              pw[y] = *reinterpret_cast<uint32_t*>(&hh);
            }
            if (p.out_aligned32) {
              st_global_v8(orow + c * 32 + x * 16, pw);
            } else {                                    // the interface only asks for 16-byte alignment
              uint4* dst = reinterpret_cast<uint4*>(orow + c * 32 + x * 16);
              dst[0] = make_uint4(pw[0], pw[1], pw[2], pw[3]);
              dst[1] = make_uint4(pw[4], pw[5], pw[6], pw[7]);
            }
          }
        }
      }
      if (warp_in_group == 0 && lane == 0) ITRACE(n_item, h ? 14 : 9);
      ++n_merge;
    } else if (row < q_rows) {
      // a query block that routed nothing in keep-or-drop mode has no attention mass at all
      for (int c = 0; c < kOutCh; c += 8) *reinterpret_cast<uint4*>(orow + c) = make_uint4(0, 0, 0, 0);
    }
    m_used = -INFINITY;
    l = 0.f;
    ++n_item;
    PROF_ADD(2)                                                                        // prof 2: whole epilogue
  }
#undef SWAIT
  if (lane == 0 && warp_in_group == 0 && h == 0) { PROF_FLUSH(3); CTATRACE(3, prof::gtimer()); }
}

template <class C, bool kFromMask>
__global__ void __launch_bounds__(kThreads, 1)
fwd_sm100_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                 const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_kc,
                 const __grid_constant__ CUtensorMap tm_vm, const Params p) {
  // (aligned by declaration and not by rounding the pointer, so that every address in it is a constant.  us, rounded / declared,
  //  24 heads x 4096 tokens, d = 128: 99.2 / 97.9, and 100.8 / 98.9 where the waits spin inline (see ptx_sm100.cuh))
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = smem_raw;
  unsigned char* sQ = base;
  unsigned char* sKV = base + C::kQBytes;
  Shared<C>& sm = *reinterpret_cast<Shared<C>*>(base + C::kQBytes + (kKStages + kVStages) * C::kTileBytes);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    sm.abort_flag = 0;
    for (int r = 0; r < kRecords; ++r) { mbar_init(&sm.rec_full[r], 1); mbar_init(&sm.rec_empty[r], kRecReaders); }
    for (int s = 0; s < kKStages; ++s) { mbar_init(&sm.k_full[s], 1); mbar_init(&sm.k_empty[s], 1); }
    for (int s = 0; s < kVStages; ++s) { mbar_init(&sm.v_full[s], 1); mbar_init(&sm.v_empty[s], 1); }
    mbar_init(&sm.q_full, 1); mbar_init(&sm.q_empty, 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(&sm.s_full[b], 1);
      mbar_init(&sm.pv_done[b], 1);
      mbar_init(&sm.p_full[0][b], 4);
      mbar_init(&sm.p_full[1][b], 4);
    }
    mbar_init(&sm.x_full, 256); mbar_init(&sm.o_free, 8);
    mbar_init(&sm.kc_full[0], 1); mbar_init(&sm.kc_full[1], 1);
    mbar_init(&sm.mma_drain[0], 1); mbar_init(&sm.mma_drain[1], 1);
    fence_mbar_init();
  }
  if (warp == kWarpProducer && lane == 0) {
    prefetch_tensormap(&tm_q); prefetch_tensormap(&tm_k); prefetch_tensormap(&tm_v);
    prefetch_tensormap(&tm_kc); prefetch_tensormap(&tm_vm);
  }
  if (warp == 0) { tmem_alloc(&sm.tmem_base, kTmemCols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;
  kernel_wait();

  if (warp < 8) {
    softmax_role<C>(sm, p, tmem, warp / 4, warp % 4, lane);
  } else if (warp == kWarpRouter) {
    router_role<C, kFromMask>(sm, p, lane);
  } else if (warp == kWarpProducer) {
    if (lane == 0) producer_role<C>(sm, p, sQ, sKV, &tm_q, &tm_k, &tm_v, &tm_kc, &tm_vm);
  } else if (warp == kWarpQK) {
    mma_qk_role<C>(sm, p, sQ, sKV, tmem);
  } else {
    mma_pv_role<C>(sm, p, sKV, tmem);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

template <class C>
cudaError_t launch_instance(const Problem& p, const Maps& m, const Params& prm, int grid, cudaStream_t stream) {
  const size_t smem = C::kQBytes + (kKStages + kVStages) * C::kTileBytes + sizeof(Shared<C>);
  // the pre-pass variant is a kernel of its own, so that the in-kernel router's code is what it is without it
  auto kernel = p.routing == SOL_ROUTING_PREPASS && p.mode != SOL_MODE_DENSE ? fwd_sm100_kernel<C, true> : fwd_sm100_kernel<C, false>;
  return launch_after(kernel, dim3(grid), kThreads, smem, smem, 0, stream, m.q, m.k, m.v, m.kc, m.vm, prm);
}

}  // namespace

long long g_wait_limit = kWaitCycles;
int g_withhold_tile = -1;

}  // namespace fwd

bool fwd_sm100_supports(const Problem& p) {
  return (p.d == 64 || p.d == 128) && p.block_q == p.block_k && (p.block_k == 64 || p.block_k == 128);
}

void fwd_sm100_set_wait(long long wait_cycles, int withhold_tile) {
  fwd::g_wait_limit = wait_cycles > 0 ? wait_cycles : ptx::kWaitCycles;
  fwd::g_withhold_tile = withhold_tile;
}

cudaError_t launch_fwd_sm100(const Problem& p, const __nv_bfloat16* q, const __nv_bfloat16* k,
                             const __nv_bfloat16* v, __nv_bfloat16* out, const WsPtrs& ws, const float* tau,
                             int32_t* counts, uint32_t* mask_out, cudaStream_t stream,
                             int* n_launches) {
  if (!fwd_sm100_supports(p)) return cudaErrorInvalidValue;
  int sms = 0;
  cudaError_t e = fwd::sm_count(&sms);
  if (e != cudaSuccess) return e;
  if (p.mode == SOL_MODE_DENSE && dense_in_pairs(p.BH, p.N, p.d, p.block_k, sms))
    return fwd::launch_dense(p, q, k, v, out, ws, counts, mask_out, sms, fwd::g_wait_limit, fwd::g_withhold_tile, stream,
                             n_launches);
  // 64-token blocks: several query blocks per CTA need more blocks than SMs.  Up to one block per SM a CTA has one in either
  // kernel, and here both softmax warpgroups share its columns.  us a call, here / there: 2 heads x 4096 tokens, d = 64 30.7 /
  // 39.9, d = 128 35.9 / 44.1; 2 x 4500, d = 64 30.0 / 37.9.
  if (p.block_k == 64 && p.mode != SOL_MODE_DENSE && (long long)p.call_heads * p.Nq > sms)
    return fwd::launch_b64(p, q, k, v, out, ws, tau, counts, mask_out, fwd::g_wait_limit, fwd::g_withhold_tile, stream,
                           n_launches);
  fwd::Maps m;
  fwd::Params prm;
  if (!fwd::prepare(p, q, k, v, out, ws, tau, counts, mask_out, p.block_k, &m, &prm)) return cudaErrorInvalidValue;
  prm.total_work = p.BH * p.Nq;
  prm.wait_limit = fwd::g_wait_limit;
  prm.withhold_tile = fwd::g_withhold_tile;
  const int grid = prm.total_work < sms ? prm.total_work : sms;
  if (p.block_k == 128)
    e = p.d == 128 ? fwd::launch_instance<fwd::Cfg<128, 128>>(p, m, prm, grid, stream)
                   : fwd::launch_instance<fwd::Cfg<64, 128>>(p, m, prm, grid, stream);
  else
    e = p.d == 128 ? fwd::launch_instance<fwd::Cfg<128, 64>>(p, m, prm, grid, stream)
                   : fwd::launch_instance<fwd::Cfg<64, 64>>(p, m, prm, grid, stream);
  if (n_launches) *n_launches += 1;
  return e;
}

}  // namespace sol
