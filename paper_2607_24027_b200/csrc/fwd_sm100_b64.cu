// Sol-Attn fused forward (Algorithm 1) for sm_100a with 64-token blocks: TMA + tcgen05.mma + TMEM.
//
// The tensor core's query tile has 128 rows at full rate (an M = 64 MMA takes as long), so one query block
// of 64 tokens per tile would leave half of the matrix and softmax work unused.  Here a persistent CTA of
// 480 threads works on up to 256 consecutive query rows of one head at a time, as two STREAMS of 128 rows,
// i.e. four query blocks.  Each stream has its own query tile, score buffers, accumulator, softmax warpgroup
// and pair of MMA-issuing warps; the two share every K and V tile that both of them need.  The query blocks route
// independently: a tile is computed for a stream when either of its two blocks wants it, the warps of a
// block that does not want it skip its softmax, and the P V MMA leaves that block's accumulator lanes alone
// (its disable-output-lane operand).  Neighbouring query blocks route much alike, so little is computed in
// vain.  24 heads x 9000 tokens, d = 64: 0.45 ms a call, where one query block per tile took 0.63 ms for this kernel alone.
//
// (With 128-token blocks, where a tile is full anyway, the same structure takes fewer cycles in dense mode
// but more energy, and the part runs at its power limit: 20.0 against 19.9 ms at 40 heads and 32 760
// tokens, and 4-6 % more in the routed modes, where two query blocks walk one list.  fwd_sm100.cu stays
// for that.)
//
// Warp roles, which talk through mbarriers:
//
//   router   (warp 8)  pulls work items from a global counter and walks the pooled keys in chunks of 64
//                      blocks.  For every key block it evaluates the proxy s_ij = scale * Qbar_i . KC_j
//                      (Eq. 3) in fp32 for each query block of the item and compares it with tau_i
//                      (Eq. 4).  The decisions only ever live in a small shared-memory record: a list of
//                      tile descriptors, each with one flag per query block, and the per-column bias of
//                      the approximate tile.  Nothing of the proxy map goes to global memory.
//   producer (warps 9 and 14, one lane each: Q and K; V) reads the records and issues TMA loads: one approximate tile per
//                      chunk (KC chunk, mean-V chunk) and K_j / V_j ONLY for key blocks that some
//                      query block of the item routed.
//   mma      (warps 10-13) two issuing warps per stream, one for the scores and one for P V, with two score
//                      buffers: the scores of a tile are computed while the one before is in its softmax.
//   softmax  (warps 0-3 and 4-7) warpgroup s serves stream s; thread = query row, with its running
//                      (m, l).  Both branches of the method update the same state: an approximate tile
//                      is an ordinary tile whose columns carry the bias log2(n_j) (Eqs. 9-10:
//                      multiplicity n_j in the denominator, mean value times n_j in the numerator) or
//                      -inf for routed / padded columns.  O is rescaled lazily, only when the running
//                      maximum grows by more than 2^8.
//
// Work item size: four query blocks share loads and tiles best, but a problem with fewer than two blocks per SM is cut into
// items of two (a stream each), so that every SM has something to do.  (One with at most one block per SM goes to
// fwd_sm100.cu.)
//
// TMEM (512 columns): stream s, score buffer x: S at 64 (2 s + x); O_s at 256 + s d.  P (bf16) of a tile
// overwrites the start of its S.
//
// Every mbarrier wait is bounded: when one expires the CTA records SOL_ERR_DEVICE_TIMEOUT in the
// workspace status word, all roles drain, TMEM is released and the kernel returns.
#include "fwd_sm100_common.cuh"

namespace sol {
namespace fwd {
namespace {

constexpr int kBlk = 64;                         // block_q = block_k = key columns of a tile
constexpr int kSub = kRowsQ / kBlk;              // query blocks per stream
constexpr int kNQ = 2 * kSub;                    // query blocks per full work item
constexpr uint32_t kSubMask = (1u << kSub) - 1;
// Ring of K tiles, and ring of V tiles.  A tile of 64 keys is 8 or 16 KB, little beside the time its copy takes: with two slots
// 312 us at 16 heads x 11 160 tokens, d = 64, keep-or-drop and 541 us at 24 x 9000, with three 312 / 540, with four 304 / 530
// (K loads four tiles ahead of V loads instead of two: 308 / 533).
constexpr int kStages = 4;
constexpr int kGroup = 16;                       // pooled keys per router staging buffer
constexpr int kRecords = 4;                      // ring of routing records
constexpr int kWarpQK = 10, kWarpPV = 12;        // one warp each per stream
constexpr int kWarpProducerV = 14;               // (warp kWarpProducer: query and K tiles)
constexpr int kThreads64 = 480;
constexpr int kTmemS = 0, kTmemO = 256;

// Compile-time shape of one kernel instance.
template <int D>
struct Cfg {
  static constexpr int kD = D;                     // head dimension
  static constexpr int kBoxes = D / 64;            // 64-channel TMA boxes per tile row
  static constexpr int kQBytes = kRowsQ * D * 2;   // a query tile
  static constexpr int kTileBytes = kBlk * D * 2;  // one K-like or V-like tile
  static constexpr int kQBoxBytes = kRowsQ * 128;  // one box of a query tile (64 channels x 128 rows)
  static constexpr int kBoxBytes = kBlk * 128;     // one box of a K-like / V-like tile
  static_assert(D == 64 || D == 128, "head dimension");
};

// The router turns every chunk of `block` key blocks into a record: a flat list of tile descriptors
// that the other roles only have to read.  A descriptor is (row coordinate << 5) | kTileApprox |
// one bit per query block of the item that uses the tile (bit u, stream u / kSub); the coordinate is the
// first key row of an exact tile or the first pooled row of an approximate one.
constexpr uint32_t kTileApprox = 16;     // approximate-branch tile (pooled keys / mean values)
constexpr int kRecFirst = 1, kRecLast = 2;   // first / last chunk of its work item

struct alignas(16) Record {
  float bias[kNQ][kBlk];        // approximate-tile column bias: log2(n_j) / (scale * log2 e), or -inf
  int32_t work;                 // work item, or -1: no more work
  int32_t b, h;                 // batch and head of the work item
  int32_t q_row[2];             // first query row of each stream
  int32_t flags;                // kRecFirst | kRecLast
  int32_t valid;                // bit u: query block u of the item exists
  int32_t n;                    // number of descriptors
  int32_t last[2];              // index of each stream's last descriptor in this record, or -1
  uint32_t desc[kBlk + 2];
};

template <class C>
struct Shared {
  float kc_stage[2][kGroup * C::kD];   // router: fp32 pooled keys being scored / the next ones
  float qbar_s[kNQ][C::kD];            // router: pooled queries of the current work item
  Record rec[kRecords];
  uint64_t rec_full[kRecords], rec_empty[kRecords];
  uint64_t k_full[kStages], k_empty[kStages], v_full[kStages], v_empty[kStages];
  // one of each per stream:
  uint64_t q_full[2], q_empty[2];
  uint64_t o_free[2];           // the accumulator of a finished work item (with a tile) has been read
  // one of each per stream and score buffer:
  uint64_t s_full[2][2];        // the scores of a tile are in TMEM
  uint64_t p_full[2][2];        // its P is in TMEM
  uint64_t pv_done[2][2];       // its P V is in the accumulator
  uint64_t kc_full[2];          // router staging buffers filled
  uint64_t mma_drain[4];        // abort path only: all MMAs issued by a role have retired
  uint32_t tmem_base;
  int abort_flag;
};

// Every role has `sm` and `wait_limit` in scope; WAIT is a bounded wait on one of its barriers.
#define WAIT(bar, parity) mbar_wait((bar), (parity), &sm.abort_flag, wait_limit)

// ------------------------------------------------------------------------------------------------
// router: one warp
// kFromMask: the decisions were taken by the routing pre-pass and are read back from the mask (one bit per
// (query block, key block)) instead of being scored here.
template <class C, bool kFromMask>
__device__ void router_role(Shared<C>& sm, const Params& p, int lane) {
  constexpr int kD = C::kD, kHalfPieces = C::kD / 8;
  constexpr uint32_t kMaskA = kSubMask, kMaskB = kSubMask << kSub;
  const unsigned full = 0xffffffffu;
  const unsigned below = (1u << lane) - 1u;
  const long long wait_limit = p.wait_limit;
  uint32_t n_rec = 0, n_copy = 0, n_use = 0;   // records written; staging copies issued / consumed
  uint32_t n_item = 0;
  const int n_chunks = ceil_div(p.Nk, kBlk);
  const int mask_words = ceil_div(p.Nk, 32);
  const float inv_sl2 = 1.f / (p.scale * 1.4426950408889634f);   // biases are stored in raw-score units
  constexpr bool from_mask = kFromMask, score = !kFromMask;
  const float bias_full = log2f((float)kBlk) * inv_sl2;                          // log2 n_j of a full block ...
  const float bias_last = log2f((float)(p.N - (p.Nk - 1) * kBlk)) * inv_sl2;     // ... and of the ragged last one
  bool alive = true;
  while (alive) {
    // the first work item is the CTA's own number (a round trip to memory less at the start), then the counter's
    int w = (int)blockIdx.x;
    if (n_item > 0) {
      if (lane == 0) w = (int)gridDim.x + atomicAdd(p.status + kStatusTileCounter, 1);
      w = __shfl_sync(full, w, 0);
    }
    if (w >= p.total_work) break;
    const int bh = w / p.items_per_head;
    const int i0 = (w - bh * p.items_per_head) * p.per_item;
    const float* kc_head = p.kc + (size_t)bh * p.Nk * kD;
    // Bulk-copy kGroup pooled keys (contiguous in memory) into a staging buffer; the copy of the next
    // ones is in flight while these are scored.
    auto stage_group = [&](int jb) {
      if (!score || jb >= p.Nk) return;
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
    stage_group(kGroup);
    // query block u of the item: the streams take one block each until a full item gives them two
    const int step = p.per_item == kNQ ? 1 : kSub;
    int valid = 0;
    float tau_u[kNQ];
    __syncwarp();
#pragma unroll
    for (int u = 0; u < kNQ; ++u) {
      const int i = i0 + u / step;
      const bool ok = u % step == 0 && u / step < p.per_item && i < p.Nq;
      valid |= (ok ? 1 : 0) << u;
      tau_u[u] = INFINITY;
      if (score) {
        // the pooled query goes to shared memory (one 16-byte piece per lane)
        if (lane < kD / 4)
          reinterpret_cast<float4*>(sm.qbar_s[u])[lane] =
              ok ? __ldg(reinterpret_cast<const float4*>(p.qbar + ((size_t)bh * p.Nq + i) * kD) + lane)
                 : make_float4(0.f, 0.f, 0.f, 0.f);
        if (ok) tau_u[u] = p.tau[(size_t)bh * p.Nq + i];
      }
    }
    __syncwarp();
    const size_t row0 = (size_t)bh * p.Nq + i0;      // counts / mask row of block u: row0 + u / step
    int count[kNQ];
#pragma unroll
    for (int u = 0; u < kNQ; ++u) count[u] = 0;
    for (int t = 0; t < n_chunks; ++t) {
      Record& rec = sm.rec[n_rec % kRecords];
      if (!WAIT(&sm.rec_empty[n_rec % kRecords], ((n_rec / kRecords) & 1) ^ 1)) {
        if (lane == 0) flag_abort(sm, p, 100);
        alive = false;
        break;
      }
      const int j0 = t * kBlk;
      uint32_t words = 0;                            // lane g * kNQ + u keeps the decisions of group g, query block u
      uint32_t approx = 0;                           // query blocks with an unselected key block in this chunk
#pragma unroll 1
      for (int g = 0; g < kBlk / 32; ++g) {
        const int jbase = j0 + g * 32;
        const int j = jbase + lane;
        float dot[kNQ];
#pragma unroll
        for (int u = 0; u < kNQ; ++u) dot[u] = 0.f;
        if (score && jbase < p.Nk) {
          // Two steps of 16 staged keys: lane l takes key l % 16 and half l / 16 of its channels.  A lane
          // starts at 16-byte piece l of its half and walks round, so that the lanes spread over the
          // shared-memory bank groups although the rows are a multiple of 128 bytes apart.
#pragma unroll 1
          for (int half = 0; half < 2; ++half) {
            const int jb = jbase + half * kGroup;
            if (jb >= p.Nk) break;
            const uint32_t buf = n_use & 1;
            if (!WAIT(&sm.kc_full[buf], (n_use >> 1) & 1)) {
              if (lane == 0) flag_abort(sm, p, 102);
              alive = false;
              break;
            }
            ++n_use;
            const float4* row = reinterpret_cast<const float4*>(sm.kc_stage[buf] + (lane % kGroup) * kD) +
                                (lane / kGroup) * kHalfPieces;
            const float4* qv = reinterpret_cast<const float4*>(sm.qbar_s[0]) + (lane / kGroup) * kHalfPieces;
            float a0[kNQ], a1[kNQ];
#pragma unroll
            for (int u = 0; u < kNQ; ++u) a0[u] = a1[u] = 0.f;
#pragma unroll 4
            for (int c = 0; c < kHalfPieces; ++c) {
              const int piece = (c + lane) & (kHalfPieces - 1);
              const float4 kk = row[piece];
#pragma unroll
              for (int u = 0; u < kNQ; ++u) {
                const float4 qq = qv[u * (kD / 4) + piece];
                a0[u] = fmaf(qq.x, kk.x, a0[u]);
                a1[u] = fmaf(qq.y, kk.y, a1[u]);
                a0[u] = fmaf(qq.z, kk.z, a0[u]);
                a1[u] = fmaf(qq.w, kk.w, a1[u]);
              }
            }
            stage_group(jb + 2 * kGroup);             // the buffer is free: the keys after next
#pragma unroll
            for (int u = 0; u < kNQ; ++u) {
              float s = a0[u] + a1[u];
              s += __shfl_xor_sync(full, s, 16);
              if (lane / kGroup == half) dot[u] = s;
            }
          }
          if (!alive) break;
        }
        const bool in_range = j < p.Nk;
        const bool is_forced = p.forced && in_range && p.forced[j];
#pragma unroll
        for (int u = 0; u < kNQ; ++u) {
          const bool exists = (valid >> u) & 1;
          bool sel;
          if (from_mask) {
            sel = exists && in_range &&
                  ((p.mask_out[(row0 + u / step) * mask_words + jbase / 32] >> lane) & 1u);
          } else {
            sel = (in_range && p.scale * dot[u] > tau_u[u]) || is_forced;
          }
          sel = sel && exists;
          const unsigned m = __ballot_sync(full, sel);
          if (lane == g * kNQ + u) words = m;
          if (exists && in_range && !sel) approx |= 1u << u;
          rec.bias[u][g * 32 + lane] = (in_range && !sel) ? (j == p.Nk - 1 ? bias_last : bias_full) : -INFINITY;
          count[u] += __popc(m);
          if (exists && p.mask_out && !from_mask && lane == 0 && jbase < p.Nk)
            p.mask_out[(row0 + u / step) * mask_words + jbase / 32] = m;
        }
      }
      if (!alive) break;
      approx = p.mode == SOL_MODE_SOL ? __reduce_or_sync(full, approx) : 0u;
      // The list: the approximate tile, then the routed key blocks in ascending order.  (Every query block
      // meets its own tiles in the same order whatever its neighbours in the item routed, so its result
      // does not depend on them.)
      int n = approx ? 1 : 0, last_a = (approx & kMaskA) ? 0 : -1, last_b = (approx & kMaskB) ? 0 : -1;
#pragma unroll
      for (int g = 0; g < kBlk / 32; ++g) {
        uint32_t a = 0, b = 0, mine = 0;
#pragma unroll
        for (int u = 0; u < kNQ; ++u) {
          const uint32_t m = __shfl_sync(full, words, g * kNQ + u);
          (u < kSub ? a : b) |= m;
          mine |= ((m >> lane) & 1u) << u;
        }
        const uint32_t any = a | b;
        if (mine) rec.desc[n + __popc(any & below)] = ((uint32_t)((j0 + g * 32 + lane) * kBlk) << 5) | mine;
        if (a) last_a = n + __popc(any & (0xffffffffu >> __clz(a))) - 1;
        if (b) last_b = n + __popc(any & (0xffffffffu >> __clz(b))) - 1;
        n += __popc(any);
      }
      if (lane == 0) {
        rec.work = w;
        rec.b = bh / p.st.H;
        rec.h = bh - rec.b * p.st.H;
        rec.q_row[0] = i0 * kBlk;
        rec.q_row[1] = (i0 + kSub / step) * kBlk;
        rec.valid = valid;
        rec.flags = (t == 0 ? kRecFirst : 0) | (t == n_chunks - 1 ? kRecLast : 0);
        if (approx) rec.desc[0] = ((uint32_t)j0 << 5) | kTileApprox | approx;
        rec.n = n;
        rec.last[0] = last_a;
        rec.last[1] = last_b;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.rec_full[n_rec % kRecords]);
      ++n_rec;
    }
    if (alive && lane == 0 && p.counts) {
#pragma unroll
      for (int u = 0; u < kNQ; ++u)
        if ((valid >> u) & 1) p.counts[row0 + u / step] = count[u];
    }
    ++n_item;
  }
  if (!alive) {
    // let staging copies that are still in flight land before the CTA's shared memory goes away
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
// producers: one thread loads the query and K tiles, another (of another warp) the V tiles.  One thread for both needs about
// 1300 cycles per tile for looking at records and slots in turn and issuing, more than anyone else here: 271 / 260 us at
// 16 heads x 11 160 tokens, d = 64, keep-or-drop.
//
// pooled = true: KC / mean-V operands, dense [B*H][Nk][d]; else q, k, v in the caller's layout.
// A tile is C::kBoxes boxes of 64 channels, each `box` bytes long in shared memory.
template <class C>
__device__ __forceinline__ void load_tile(const Params& p, uint32_t bytes, int box, const CUtensorMap* tm, uint64_t* full,
                                          unsigned char* dst, int row, int b, int h, bool pooled) {
  mbar_arrive_expect_tx(full, bytes);
  const bool rows_inner = pooled || p.rows_inner;
  const int c1 = rows_inner ? row : h, c2 = rows_inner ? h : row;
  tma_load_4d(dst, tm, full, 0, c1, c2, b);
  if constexpr (C::kBoxes == 2) tma_load_4d(dst + box, tm, full, 64, c1, c2, b);
}
#define NEED(bar, parity) if (!WAIT(bar, parity)) { ok = false; break; }

template <class C>
__device__ void qk_producer_role(Shared<C>& sm, const Params& p, unsigned char* sQ, unsigned char* sKV,
                                 const CUtensorMap* tm_q, const CUtensorMap* tm_k, const CUtensorMap* tm_kc) {
  const long long wait_limit = p.wait_limit;
  uint32_t n = 0, n_q[2] = {0, 0};             // K tiles and query tiles so far
  bool ok = true;
  for (uint32_t n_rec = 0; ok; ++n_rec) {
    const uint32_t r = n_rec % kRecords;
    NEED(&sm.rec_full[r], (n_rec / kRecords) & 1)
    const Record& rec = sm.rec[r];
    if (rec.work < 0) break;
    const int n_desc = rec.n, b = rec.b, h = rec.h;
    if (rec.flags & kRecFirst) {
      // Q of both streams, once per work item.  A slot frees when the stream's last score GEMM of the
      // previous item retires.
#pragma unroll
      for (int s = 0; s < 2; ++s) {
        if (!((rec.valid >> (s * kSub)) & 1)) continue;
        NEED(&sm.q_empty[s], (n_q[s] & 1) ^ 1)
        load_tile<C>(p, C::kQBytes, C::kQBoxBytes, tm_q, &sm.q_full[s], sQ + s * C::kQBytes, rec.q_row[s], b, h, false);
        ++n_q[s];
      }
      if (!ok) break;
    }
    for (int e = 0; e < n_desc; ++e, ++n) {
      const uint32_t d = rec.desc[e], s = n % kStages;
      NEED(&sm.k_empty[s], ((n / kStages) & 1) ^ 1)
      load_tile<C>(p, C::kTileBytes, C::kBoxBytes, (d & kTileApprox) ? tm_kc : tm_k, &sm.k_full[s],
                   sKV + (size_t)s * C::kTileBytes, (int)(d >> 5), b, h, (d & kTileApprox) != 0);
    }
    if (ok) mbar_arrive(&sm.rec_empty[r]);
  }
  if (!ok) flag_abort(sm, p, 200);
  // The consumers wait for every K, V and Q tile of a normal run; after an abort, let copies that are
  // still in flight land before the CTA's shared memory goes away.
  if (sm.abort_flag) {
    int never = 0;                             // this drain must not be cut short by the abort flag
    for (int s = 0; s < 2; ++s)
      if (n_q[s] > 0) mbar_wait(&sm.q_full[s], (n_q[s] - 1) & 1, &never, wait_limit);
    for (uint32_t back = 1; back <= kStages && back <= n; ++back)
      mbar_wait(&sm.k_full[(n - back) % kStages], ((n - back) / kStages) & 1, &never, wait_limit);
  }
}

template <class C>
__device__ void v_producer_role(Shared<C>& sm, const Params& p, unsigned char* sKV, const CUtensorMap* tm_v,
                                const CUtensorMap* tm_vm) {
  const long long wait_limit = p.wait_limit;
  uint32_t n = 0;
  bool ok = true;
  for (uint32_t n_rec = 0; ok; ++n_rec) {
    const uint32_t r = n_rec % kRecords;
    NEED(&sm.rec_full[r], (n_rec / kRecords) & 1)
    const Record& rec = sm.rec[r];
    if (rec.work < 0) break;
    const int n_desc = rec.n, b = rec.b, h = rec.h;
    for (int e = 0; e < n_desc; ++e, ++n) {
      const uint32_t d = rec.desc[e], s = n % kStages;
      NEED(&sm.v_empty[s], ((n / kStages) & 1) ^ 1)
      load_tile<C>(p, C::kTileBytes, C::kBoxBytes, (d & kTileApprox) ? tm_vm : tm_v, &sm.v_full[s],
                   sKV + (size_t)(kStages + s) * C::kTileBytes, (int)(d >> 5), b, h, (d & kTileApprox) != 0);
    }
    if (ok) mbar_arrive(&sm.rec_empty[r]);
  }
  if (!ok) flag_abort(sm, p, 201);
  if (sm.abort_flag) {
    int never = 0;
    for (uint32_t back = 1; back <= kStages && back <= n; ++back)
      mbar_wait(&sm.v_full[(n - back) % kStages], ((n - back) / kStages) & 1, &never, wait_limit);
  }
}
#undef NEED

// ------------------------------------------------------------------------------------------------
// Two issuing warps per stream s, one for the score GEMMs and one for the value GEMMs.  A warp that did both had to look at
// every barrier in turn without ever sleeping (each side may have something to release that the other waits for): 304 us at
// 16 heads x 11 160 tokens, d = 64, keep-or-drop, where two that simply wait take 271, although a score GEMM now needs
// a completion signal of the P V whose buffer it takes over.
//
// The warps run in lockstep and one elected lane issues: with warp-uniform control flow and operands the
// compiler keeps descriptors and addresses in uniform registers, where the MMA instruction wants them.
// Every wait is made uniform by a vote; a lane that fell behind could otherwise miss a phase.
//
// A tile that only the other stream uses is released as soon as it has landed (not earlier: an arrival
// before that could be taken for one of the slot's previous tile).
#define NEED(bar, parity) if (!__all_sync(0xffffffffu, WAIT(bar, parity))) { ok = false; break; }

// Abort path: TMEM must not be released while MMAs are still writing to it, so the role asks for a
// completion signal behind everything it has issued and waits for it (bounded).
template <class C>
__device__ void drain_mmas(Shared<C>& sm, const Params& p, bool ok, bool leader, int which) {
  if (!ok && leader) flag_abort(sm, p, 300 + which);
  __syncwarp();
  if (sm.abort_flag) {
    if (leader) mma_commit(&sm.mma_drain[which]);
    int never = 0;
    mbar_wait(&sm.mma_drain[which], 0, &never, p.wait_limit);
  }
}

// S = Q K^T of the stream's tiles, alternating between its two score buffers
template <class C>
__device__ void mma_qk_role(Shared<C>& sm, const Params& p, unsigned char* sQ, unsigned char* sKV, uint32_t tmem, int s) {
  constexpr int kD = C::kD, kTileBytes = C::kTileBytes;
  const long long wait_limit = p.wait_limit;
  const uint32_t idesc_qk = make_idesc_bf16(kRowsQ, kBlk, false, false);
  const uint32_t q_lo = (smem_addr(sQ + s * C::kQBytes) >> 4) | (1u << 16);
  const uint32_t k_lo0 = (smem_addr(sKV) >> 4) | (1u << 16);
  const uint32_t t_s0 = tmem + kTmemS + s * 2 * kBlk;
  const bool leader = elect_one();
  uint32_t slot = 0, par = 0, n_item = 0, n = 0;   // ring position; work items with the stream; tiles issued
  bool fresh = false, ok = true;               // the work item's Q has not been waited for
  for (uint32_t n_rec = 0; ok; ++n_rec) {
    const uint32_t r = n_rec % kRecords;
    NEED(&sm.rec_full[r], (n_rec / kRecords) & 1)
    const Record& rec = sm.rec[r];
    if (rec.work < 0) break;
    const int n_desc = rec.n, last = rec.last[s];
    const bool exists = (rec.valid >> (s * kSub)) & 1, last_chunk = (rec.flags & kRecLast) != 0;
    if (exists && (rec.flags & kRecFirst)) { fresh = true; ++n_item; }
    for (int e = 0; e < n_desc; ++e) {
      const uint32_t use = (rec.desc[e] >> (s * kSub)) & kSubMask;
      NEED(&sm.k_full[slot], par)
      if (use) {
        if (fresh) { NEED(&sm.q_full[s], (n_item - 1) & 1) }
        fresh = false;
        const uint32_t x = n & 1;
        // P overwrites S: the P V of the buffer's tile before must have read P
        if (n >= 2) { NEED(&sm.pv_done[s][x], ((n - 2) >> 1) & 1) }
        tc_fence_after();
        const uint32_t k_lo = k_lo0 + slot * (kTileBytes >> 4);
#pragma unroll
        for (int ks = 0; ks < kD / 16; ++ks) {
          // K-step ks: 16 channels = 32 bytes inside box ks / 4
          const uint32_t off_q = ((ks / 4) * C::kQBoxBytes + (ks % 4) * 32) >> 4;
          const uint32_t off_k = ((ks / 4) * C::kBoxBytes + (ks % 4) * 32) >> 4;
          const uint64_t da = desc_from_lo(q_lo + off_q), db = desc_from_lo(k_lo + off_k);
          if (leader) mma_ss(t_s0 + x * kBlk, da, db, idesc_qk, ks > 0);
        }
        if (leader) {
          mma_commit(&sm.s_full[s][x]);
          mma_commit(&sm.k_empty[slot]);
          if (last_chunk && e == last) mma_commit(&sm.q_empty[s]);
        }
        ++n;
      } else if (leader) {
        mbar_arrive(&sm.k_empty[slot]);
      }
      if (++slot == kStages) { slot = 0; par ^= 1; }
    }
    if (!ok) break;
    if (exists && last_chunk && last < 0) {    // an item without a tile in its last chunk hands Q back here
      if (fresh) {                             // nothing has read Q
        NEED(&sm.q_full[s], (n_item - 1) & 1)
        if (leader) mbar_arrive(&sm.q_empty[s]);
        fresh = false;
      } else if (leader) {
        mma_commit(&sm.q_empty[s]);
      }
    }
    __syncwarp();
    if (leader) mbar_arrive(&sm.rec_empty[r]);
  }
  drain_mmas(sm, p, ok, leader, s);
}

// O (+)= P V of the stream's tiles
template <class C>
__device__ void mma_pv_role(Shared<C>& sm, const Params& p, unsigned char* sKV, uint32_t tmem, int s) {
  constexpr int kD = C::kD, kTileBytes = C::kTileBytes;
  const long long wait_limit = p.wait_limit;
  const uint32_t idesc_pv = make_idesc_bf16(kRowsQ, kD, false, true);
  // V is the MN-major operand: its 64-channel boxes are C::kBoxBytes apart (leading offset), groups of
  // 8 key rows 1024 bytes apart; a K-step of 16 keys advances the start by 2048 bytes.
  const uint32_t v_lo0 = (smem_addr(sKV + kStages * kTileBytes) >> 4) | ((uint32_t)(C::kBoxBytes >> 4) << 16);
  const uint32_t t_s0 = tmem + kTmemS + s * 2 * kBlk, t_o = tmem + kTmemO + s * kD;
  const bool leader = elect_one();
  uint32_t slot = 0, par = 0, n = 0;
  uint32_t n_acc = 0;                          // work items with a tile of the stream
  uint32_t started = 0;                        // query blocks of the stream whose accumulator holds something
  bool fresh = false, ok = true;
  for (uint32_t n_rec = 0; ok; ++n_rec) {
    const uint32_t r = n_rec % kRecords;
    NEED(&sm.rec_full[r], (n_rec / kRecords) & 1)
    const Record& rec = sm.rec[r];
    if (rec.work < 0) break;
    const int n_desc = rec.n;
    if (((rec.valid >> (s * kSub)) & 1) && (rec.flags & kRecFirst)) fresh = true;
    for (int e = 0; e < n_desc; ++e) {
      const uint32_t use = (rec.desc[e] >> (s * kSub)) & kSubMask;
      NEED(&sm.v_full[slot], par)
      if (use) {
        if (fresh) {
          // the first P V of a work item overwrites O: the epilogue of the last item with a tile must have read it
          if (n_acc > 0) { NEED(&sm.o_free[s], (n_acc - 1) & 1) }
          started = 0;
          ++n_acc;
        }
        fresh = false;
        const uint32_t x = n & 1;
        NEED(&sm.p_full[s][x], (n >> 1) & 1)
        tc_fence_after();
        const uint32_t v_lo = v_lo0 + slot * (kTileBytes >> 4);
        // lanes of a query block that does not use the tile are left alone; a block's first tile overwrites
        const uint32_t first = use & ~started, more = use & started;
        const uint32_t a_p0 = t_s0 + x * kBlk;
#pragma unroll
        for (int ks = 0; ks < kBlk / 16; ++ks) {
          const uint64_t dv = desc_from_lo(v_lo + ((ks * 2048) >> 4));
          if (more && leader)
            mma_ts_lanes(t_o, a_p0 + ks * 8, dv, idesc_pv, 1u, (more & 1) ? 0u : ~0u, (more & 2) ? 0u : ~0u);
          if (first && leader)
            mma_ts_lanes(t_o, a_p0 + ks * 8, dv, idesc_pv, ks > 0, (first & 1) ? 0u : ~0u, (first & 2) ? 0u : ~0u);
        }
        started |= use;
        if (leader) {
          mma_commit(&sm.pv_done[s][x]);
          // (test hook: a withheld completion signal makes the bounded waits on it run out)
          if (s != 0 || (int)n != p.withhold_tile) mma_commit(&sm.v_empty[slot]);
        }
        ++n;
      } else if (leader) {
        mbar_arrive(&sm.v_empty[slot]);
      }
      if (++slot == kStages) { slot = 0; par ^= 1; }
    }
    if (!ok) break;
    __syncwarp();
    if (leader) mbar_arrive(&sm.rec_empty[r]);
  }
  drain_mmas(sm, p, ok, leader, 2 + s);
}
#undef NEED

// ------------------------------------------------------------------------------------------------
// softmax + correction + epilogue: one warpgroup of 128 threads per stream; thread = query row.
template <class C>
__device__ void softmax_role(Shared<C>& sm, const Params& p, uint32_t tmem, int s, int warp_in_group, int lane) {
  constexpr int kD = C::kD;
  const unsigned full = 0xffffffffu;
  const long long wait_limit = p.wait_limit;
  const uint32_t lane_base = tmem + ((uint32_t)(warp_in_group * 32) << 16);
  const uint32_t t_s0 = lane_base + kTmemS + s * 2 * kBlk;
  const uint32_t t_o = lane_base + kTmemO + s * kD;
  const int row = warp_in_group * 32 + lane;                 // row of the query tile
  const int u = s * kSub + row / kBlk;                       // query block of the item (the same for a whole warp)
  const float sl2 = p.scale * 1.4426950408889634f;
  uint32_t g = 0, n_rec = 0;                                 // tiles and records so far
  uint32_t g_item0 = 0;                                      // first tile of the work item
  float m_used = -INFINITY, l = 0.f;
  bool started = false;
  // A wait that gives up must give up for the whole warp: the loop holds warp-synchronising
  // operations (TMEM loads and stores, votes), so the lanes leave together or not at all.
#define SWAIT(bar, parity) __all_sync(full, WAIT(bar, parity))
  for (;;) {
    const uint32_t r = n_rec % kRecords;
    if (!SWAIT(&sm.rec_full[r], (n_rec / kRecords) & 1)) { flag_abort(sm, p, 400); break; }
    const Record& rec = sm.rec[r];
    if (rec.work < 0) break;
    const int n = rec.n, flags = rec.flags;
    const bool exists = (rec.valid >> (s * kSub)) & 1;       // the stream has a query tile in this item
    if (flags & kRecFirst) {
      m_used = -INFINITY;
      l = 0.f;
      started = false;
      g_item0 = g;
    }
    bool ok = true;
    for (int e = 0; e < n; ++e) {
      const uint32_t dsc = rec.desc[e];
      if (!((dsc >> (s * kSub)) & kSubMask)) continue;       // a tile of the other stream
      const bool approx = (dsc & kTileApprox) != 0;
      const int cols_valid = approx ? kBlk : min(kBlk, p.N - (int)(dsc >> 5));
      const bool general = approx || cols_valid < kBlk;
      const uint32_t x = g & 1;
      const uint32_t t_s = t_s0 + x * kBlk;
      // (no vote on this wait, the one wait of every tile: the 32 lanes poll the same barrier, abort flag
      //  and clock in lockstep and leave the loop together; the rarer waits are made uniform by a vote)
      if (!WAIT(&sm.s_full[s][x], (g >> 1) & 1)) { flag_abort(sm, p, 401); ok = false; break; }
      tc_fence_after();
      if (!((dsc >> u) & 1)) {
        // this warp's query block does not use the tile: its P is never read into its accumulator
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.p_full[s][x]);
        ++g;
        continue;
      }
      // ---- this row of S (64 fp32) into registers with one wait
      uint32_t sr[kBlk];
      tmem_ld_cols<kBlk>(t_s, sr);
      tmem_ld_wait();
      if (general) {
        // bring the rare tiles (approximate chunk, ragged last block) to the common form
        // logit = sl2 * x by folding the column bias into x; -inf marks masked columns
        if (approx) {
          const float4* bias4 = reinterpret_cast<const float4*>(&rec.bias[u][0]);
#pragma unroll
          for (int c = 0; c < kBlk / 4; ++c) {
            const float4 bb = bias4[c];
            sr[4 * c] = __float_as_uint(__uint_as_float(sr[4 * c]) + bb.x);
            sr[4 * c + 1] = __float_as_uint(__uint_as_float(sr[4 * c + 1]) + bb.y);
            sr[4 * c + 2] = __float_as_uint(__uint_as_float(sr[4 * c + 2]) + bb.z);
            sr[4 * c + 3] = __float_as_uint(__uint_as_float(sr[4 * c + 3]) + bb.w);
          }
        } else {
#pragma unroll
          for (int c = 0; c < kBlk; ++c)
            if (c >= cols_valid) sr[c] = __float_as_uint(-INFINITY);
        }
      }
      float mx;
      {
        constexpr int kQ = kBlk / 4;
        float m0 = -INFINITY, m1 = -INFINITY, m2 = -INFINITY, m3 = -INFINITY;
#pragma unroll
        for (int c = 0; c < kQ; ++c) {
          m0 = fmaxf(m0, __uint_as_float(sr[c]));
          m1 = fmaxf(m1, __uint_as_float(sr[kQ + c]));
          m2 = fmaxf(m2, __uint_as_float(sr[2 * kQ + c]));
          m3 = fmaxf(m3, __uint_as_float(sr[3 * kQ + c]));
        }
        mx = fmaxf(fmaxf(m0, m1), fmaxf(m2, m3)) * sl2;     // -inf when every column is masked
      }
      // ---- running maximum, lazy rescale of O
      if (!started) {
        m_used = mx;
        started = true;
      } else if (__any_sync(full, mx > m_used + kRescaleThreshold)) {
        const float m_new = fmaxf(m_used, mx);
        const float f = (m_new == -INFINITY) ? 1.f : ex2(m_used - m_new);
        // P V of the previous tile must have landed in O
        if (!SWAIT(&sm.pv_done[s][x ^ 1], ((g - 1) >> 1) & 1)) { flag_abort(sm, p, 402); ok = false; break; }
        tc_fence_after();
#pragma unroll 1
        for (int c = 0; c < kD / 32; ++c) {
          uint32_t o[32];
          tmem_ld_32x32b_x32(t_o + c * 32, o);
          tmem_ld_wait();
#pragma unroll
          for (int y = 0; y < 32; ++y) o[y] = __float_as_uint(__uint_as_float(o[y]) * f);
          tmem_st_32x32b_x32(t_o + c * 32, o);
        }
        l *= f;
        m_used = m_new;
      }
      // ---- P = exp2(sl2 * S - m) (scaled as packed fp32 pairs); P (bf16) back to TMEM over the start of the
      //      scores.  The row sum is that of the rounded P, the weights that P V uses.  A row has one maximum here,
      //      where fwd_sm100.cu has one per column half and with it two exact weights; with the sum of the unrounded
      //      P the error against 64 bits grows from 1.80e-3 to 1.85e-3 (16 heads, d = 64, 11 160 tokens, density
      //      0.20, keep-or-drop), with this one it is 1.78e-3.
      {
        const float nm = (m_used == -INFINITY) ? 0.f : -m_used;   // a row that has seen nothing yet: all P = 0
        const float2 sl2_2 = make_float2(sl2, sl2), nm2 = make_float2(nm, nm);
        float2 s_a = make_float2(0.f, 0.f), s_b = make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < kBlk; c += 4) {
          const float2 xa = __ffma2_rn(make_float2(__uint_as_float(sr[c]), __uint_as_float(sr[c + 1])), sl2_2, nm2);
          const float2 xb = __ffma2_rn(make_float2(__uint_as_float(sr[c + 2]), __uint_as_float(sr[c + 3])), sl2_2, nm2);
          const float2 ea = make_float2(ex2(xa.x), ex2(xa.y));
          const float2 eb = make_float2(ex2(xb.x), ex2(xb.y));
          __nv_bfloat162 lo = __floats2bfloat162_rn(ea.x, ea.y);
          __nv_bfloat162 hi = __floats2bfloat162_rn(eb.x, eb.y);
          sr[c / 2] = *reinterpret_cast<uint32_t*>(&lo);
          sr[c / 2 + 1] = *reinterpret_cast<uint32_t*>(&hi);
          s_a = add_bf16x2(s_a, sr[c / 2]);
          s_b = add_bf16x2(s_b, sr[c / 2 + 1]);
        }
        const float2 t = __fadd2_rn(s_a, s_b);
        l += t.x + t.y;
        tmem_st_32x32b_x32(t_s, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();                                // one arrival per warp: 4 instead of 128 on the barrier
      if (lane == 0) mbar_arrive(&sm.p_full[s][x]);
      ++g;
    }
    if (!ok) break;
    if (exists && (flags & kRecLast)) {
      // ---- end of the work item: O / l
      const int q_row = rec.q_row[s];
      const int q_end = min(p.N, q_row + (((rec.valid >> (s * kSub + kSub - 1)) & 1) ? kRowsQ : kBlk));
      __nv_bfloat16* orow = p.out + (size_t)rec.b * (size_t)p.st.batch + (size_t)rec.h * (size_t)p.st.head +
                            (size_t)(q_row + row) * (size_t)p.st.row;
      const bool store = q_row + row < q_end;
      // the last P V of the item
      if (g != g_item0 && !SWAIT(&sm.pv_done[s][(g - 1) & 1], ((g - 1) >> 1) & 1)) {
        flag_abort(sm, p, 403);
        break;
      }
      tc_fence_after();
      // a query block that routed nothing in keep-or-drop mode, or a row without any finite logit, has no
      // attention mass at all: zero, whatever the accumulator holds
      const bool mass = m_used != -INFINITY;
      const float inv = 1.f / l;
#pragma unroll 1
      for (int c = 0; c < kD / 32; ++c) {
        uint32_t a[32];
        tmem_ld_32x32b_x32(t_o + c * 32, a);
        tmem_ld_wait();
        if (c == kD / 32 - 1) {
          // the accumulator is in registers: the next item's first P V may overwrite it
          tc_fence_before();
          __syncwarp();
          if (lane == 0 && g != g_item0) mbar_arrive(&sm.o_free[s]);   // (nothing waits for an item without tiles)
        }
        if (store) {
#pragma unroll
          for (int x = 0; x < 2; ++x) {                 // 32 bytes (16 channels) per store
            uint32_t pw[8];
#pragma unroll
            for (int y = 0; y < 8; ++y) {
              const int e0 = x * 16 + 2 * y;
              const float v0 = mass ? __uint_as_float(a[e0]) * inv : 0.f;
              const float v1 = mass ? __uint_as_float(a[e0 + 1]) * inv : 0.f;
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
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&sm.rec_empty[r]);
    ++n_rec;
  }
#undef SWAIT
}

template <class C, bool kFromMask>
__global__ void __launch_bounds__(kThreads64, 1)
fwd_sm100_b64_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                 const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_kc,
                 const __grid_constant__ CUtensorMap tm_vm, const Params p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];   // (see fwd_sm100.cu)
  unsigned char* base = smem_raw;
  unsigned char* sQ = base;
  unsigned char* sKV = base + 2 * C::kQBytes;
  Shared<C>& sm = *reinterpret_cast<Shared<C>*>(base + 2 * C::kQBytes + 2 * kStages * C::kTileBytes);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    sm.abort_flag = 0;
    // a record is released by the two producers, the four MMA warps and the 8 softmax warps
    for (int r = 0; r < kRecords; ++r) { mbar_init(&sm.rec_full[r], 1); mbar_init(&sm.rec_empty[r], 14); }
    for (int i = 0; i < kStages; ++i) {                      // a tile is released by both MMA warps
      mbar_init(&sm.k_full[i], 1); mbar_init(&sm.k_empty[i], 2);
      mbar_init(&sm.v_full[i], 1); mbar_init(&sm.v_empty[i], 2);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sm.q_full[s], 1); mbar_init(&sm.q_empty[s], 1);
      mbar_init(&sm.o_free[s], 4);
      for (int x = 0; x < 2; ++x) {
        mbar_init(&sm.s_full[s][x], 1); mbar_init(&sm.p_full[s][x], 4); mbar_init(&sm.pv_done[s][x], 1);
      }
      mbar_init(&sm.kc_full[s], 1);
      mbar_init(&sm.mma_drain[s], 1); mbar_init(&sm.mma_drain[2 + s], 1);
    }
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
    if (lane == 0) qk_producer_role<C>(sm, p, sQ, sKV, &tm_q, &tm_k, &tm_kc);
  } else if (warp == kWarpProducerV) {
    if (lane == 0) v_producer_role<C>(sm, p, sKV, &tm_v, &tm_vm);
  } else if (warp < kWarpPV) {
    mma_qk_role<C>(sm, p, sQ, sKV, tmem, warp - kWarpQK);
  } else {
    mma_pv_role<C>(sm, p, sKV, tmem, warp - kWarpPV);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

template <class C>
cudaError_t launch_instance(const Problem& p, const Maps& m, const Params& prm, int grid, cudaStream_t stream) {
  const size_t smem = 2 * C::kQBytes + 2 * kStages * C::kTileBytes + sizeof(Shared<C>);
  auto kernel = p.routing == SOL_ROUTING_PREPASS ? fwd_sm100_b64_kernel<C, true> : fwd_sm100_b64_kernel<C, false>;
  return launch_after(kernel, dim3(grid), kThreads64, smem, smem, 0, stream, m.q, m.k, m.v, m.kc, m.vm, prm);
}

}  // namespace

cudaError_t launch_b64(const Problem& p, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                       __nv_bfloat16* out, const WsPtrs& ws, const float* tau, int32_t* counts, uint32_t* mask_out,
                       long long wait_limit, int withhold_tile, cudaStream_t stream, int* n_launches) {
  Maps m;
  Params prm;
  if (!prepare(p, q, k, v, out, ws, tau, counts, mask_out, kBlk, &m, &prm)) return cudaErrorInvalidValue;
  prm.wait_limit = wait_limit;
  prm.withhold_tile = withhold_tile;
  int sms = 0;
  cudaError_t e = sm_count(&sms);
  if (e != cudaSuccess) return e;
  // as many query blocks per work item as still leave every SM one
  const long long blocks = (long long)p.BH * p.Nq;
  prm.per_item = blocks <= 2LL * sms ? 2 : kNQ;
  prm.items_per_head = ceil_div(p.Nq, prm.per_item);
  prm.total_work = p.BH * prm.items_per_head;
  const int grid = prm.total_work < sms ? prm.total_work : sms;
  e = p.d == 64 ? launch_instance<Cfg<64>>(p, m, prm, grid, stream) : launch_instance<Cfg<128>>(p, m, prm, grid, stream);
  if (n_launches) *n_launches += 1;
  return e;
}

}  // namespace fwd
}  // namespace sol
