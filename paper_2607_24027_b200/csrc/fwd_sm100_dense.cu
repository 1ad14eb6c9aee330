// Dense attention (SOL_MODE_DENSE, Eq. 1) for sm_100a, two query tiles per SM: TMA + tcgen05.mma + TMEM.
//
// Nothing is routed, so two query tiles of 128 rows can walk the same keys in step: a CTA owns 256 query rows
// of one head, and every K / V tile it loads feeds both.  That halves what an SM has to take in by TMA (51.5
// bytes per clock at most, measured: the 64 KB of a K / V pair cost 1273 cycles, more than the 1024 tensor cycles
// one query tile does with them), and it keeps the tensor core and the special-function units busy at the
// same time: one warp issues for both tiles A and B in turn,
//   P V (A, t)  Q K^T (A, t + 1)  |  P V (B, t)  Q K^T (B, t + 1)  |  ...
// so while A's GEMMs run, B's warpgroup has the special-function units to itself, and the other way round.  The
// strict order is what holds the two half a period apart.  (An issuing warp per tile lets the tensor core
// alternate between them; the exponentials of both then collide: 2425 instead of 1630 cycles of softmax per tile.
// One warp that polls for whichever is ready loses more in polling than it gains.)
//
//   softmax  (warps 0-3: tile A, 4-7: tile B) thread = query row with all 128 scores of a tile in registers;
//            P (bf16) goes back over the start of S in two halves, so that P V starts on the first while the
//            second is in its exponentials.  O is rescaled lazily (running maximum grown by more than 2^8).
//   mma      (warp 8), producer (warp 9, one lane), counts and debug mask (warp 10).
//
// TMEM: S_A [0, 128)  S_B [128, 256)  O_A [256, 256 + d)  O_B [256 + d, 256 + 2 d).
//
// 40 heads x 32 760 tokens, d = 128: 19.9 ms against 20.0 ms with one query tile per CTA (19.7 with the row sum of the
// unrounded weights, see softmax_role; the part is at its 1 kW limit in all three); d = 64, 40 x 16 000: 3.69 ms against
// 3.93 ms.  A pair of tiles takes 3 460 cycles, of which the tensor core needs 2 048: a tile's softmax, P V and next Q K^T
// follow one another, and beside the other tile's the three take that long.
// Every wait is bounded, as in the other kernels.
#include <atomic>

#include "fwd_sm100_common.cuh"

namespace sol {
namespace fwd {
namespace {

constexpr int kCols = 128;                       // keys per tile
constexpr int kSlots = 5;                        // ring of K and V tiles: K0 V0 K1 V1 ...
constexpr int kWarpMma = 8, kWarpCounts = 10;
constexpr int kTmemS = 0, kTmemO = 256;
constexpr int kRegsSoftmax = 200, kRegsOther = 104, kRegsLaunch = 168;   // registers per thread of the roles, and at launch
static_assert(8 * kRegsSoftmax + 4 * kRegsOther <= 12 * kRegsLaunch, "a warpgroup would wait for registers without end");

template <int D>
struct Cfg {
  static constexpr int kTileBytes = kCols * D * 2;         // a query, K or V tile
  static constexpr int kBoxBytes = kCols * 128;            // 64 channels of it
};

struct Shared {
  uint64_t q_full[2], q_empty[2];                // per query tile
  uint64_t kv_full[kSlots], kv_empty[kSlots];
  uint64_t s_full[2];                            // scores of a tile are in TMEM
  uint64_t p_full[2][2];                         // first / second half of the columns of P are in TMEM
  uint64_t o_full[2], o_free[2];                 // accumulator complete / read
  uint64_t mma_drain;                            // abort path only
  uint32_t tmem_base;
  int abort_flag;
};

#define WAIT(bar, parity) mbar_wait_inline((bar), (parity), &sm.abort_flag, p.wait_limit)
#define WAIT_ALL(bar, parity) __all_sync(0xffffffffu, WAIT(bar, parity))

// Work items are dealt out round robin: they all cost the same.
struct Item { int b, h, row; };
__device__ __forceinline__ Item item_at(const Params& p, int w) {
  const int bh = w / p.items_per_head;
  Item it;
  it.b = bh / p.st.H;
  it.h = bh - it.b * p.st.H;
  it.row = (w - bh * p.items_per_head) * 2 * kRowsQ;
  return it;
}

template <int D>
__device__ void producer_role(Shared& sm, const Params& p, unsigned char* sQ, unsigned char* sKV, const CUtensorMap* tm_q,
                              const CUtensorMap* tm_k, const CUtensorMap* tm_v) {
  using C = Cfg<D>;
  const int n_tiles = ceil_div(p.N, kCols);
  uint32_t m = 0, n_item = 0, n_q[2] = {0, 0};   // K / V tiles, work items and query tiles so far
  auto load = [&](const CUtensorMap* tm, uint64_t* full, unsigned char* dst, int row, const Item& it) {
    mbar_arrive_expect_tx(full, C::kTileBytes);
    const int c1 = p.rows_inner ? row : it.h, c2 = p.rows_inner ? it.h : row;
    tma_load_4d(dst, tm, full, 0, c1, c2, it.b);
    if constexpr (D == 128) tma_load_4d(dst + C::kBoxBytes, tm, full, 64, c1, c2, it.b);
  };
  bool ok = true;
  for (int w = blockIdx.x; ok && w < p.total_work; w += gridDim.x, ++n_item) {
    const Item it = item_at(p, w);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if (!WAIT(&sm.q_empty[s], (n_item & 1) ^ 1)) { ok = false; break; }
      load(tm_q, &sm.q_full[s], sQ + s * C::kTileBytes, it.row + s * kRowsQ, it);
      ++n_q[s];
      // K0 between the two, so that A's first scores do not wait for B's queries
      if (s == 0 && ok) {
        const uint32_t slot = m % kSlots;
        if (!WAIT(&sm.kv_empty[slot], ((m / kSlots) & 1) ^ 1)) { ok = false; break; }
        load(tm_k, &sm.kv_full[slot], sKV + slot * C::kTileBytes, 0, it);
        ++m;
      }
    }
    for (int x = 1; ok && x < 2 * n_tiles; ++x) {
      const uint32_t slot = m % kSlots;
      if (!WAIT(&sm.kv_empty[slot], ((m / kSlots) & 1) ^ 1)) { ok = false; break; }
      load((x & 1) ? tm_v : tm_k, &sm.kv_full[slot], sKV + slot * C::kTileBytes, (x / 2) * kCols, it);
      ++m;
    }
  }
  if (!ok) flag_abort(sm, p, 200);
  if (sm.abort_flag) {
    // let copies that are still in flight land before the CTA's shared memory goes away (not cut short by the flag)
    int never = 0;
    for (int s = 0; s < 2; ++s)
      if (n_q[s] > 0) mbar_wait_inline(&sm.q_full[s], (n_q[s] - 1) & 1, &never, p.wait_limit);
    for (uint32_t back = 0; back < kSlots && back < m; ++back) {
      const uint32_t n = m - 1 - back;
      mbar_wait_inline(&sm.kv_full[n % kSlots], (n / kSlots) & 1, &never, p.wait_limit);
    }
  }
}

template <int D>
__device__ void mma_role(Shared& sm, const Params& p, unsigned char* sQ, unsigned char* sKV, uint32_t tmem) {
  using C = Cfg<D>;
  const int n_tiles = ceil_div(p.N, kCols);
  const uint32_t idesc_qk = make_idesc_bf16(kRowsQ, kCols, false, false);
  const uint32_t idesc_pv = make_idesc_bf16(kRowsQ, D, false, true);
  const uint32_t q_lo0 = (smem_addr(sQ) >> 4) | (1u << 16);
  const uint32_t k_lo0 = (smem_addr(sKV) >> 4) | (1u << 16);
  const uint32_t v_lo0 = (smem_addr(sKV) >> 4) | ((uint32_t)(C::kBoxBytes >> 4) << 16);   // MN-major: see below
  const bool leader = elect_one();
  uint32_t m = 0, g = 0, n_item = 0;             // ring position of the current K tile; tiles and items so far
  bool ok = true;
  // S_s = Q_s K^T from ring slot `slot`
  auto scores = [&](int s, uint32_t slot) {
    const uint32_t k_lo = k_lo0 + slot * (C::kTileBytes >> 4), q_lo = q_lo0 + s * (C::kTileBytes >> 4);
    tc_fence_after();
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {        // 16 channels = 32 bytes inside box ks / 4
      const uint32_t off = ((ks / 4) * C::kBoxBytes + (ks % 4) * 32) >> 4;
      if (leader) mma_ss(tmem + kTmemS + s * kCols, desc_from_lo(q_lo + off), desc_from_lo(k_lo + off), idesc_qk, ks > 0);
    }
    if (leader) mma_commit(&sm.s_full[s]);
  };
  // half of O_s (+)= P_s V: V is the MN-major operand, its 64-channel boxes are kBoxBytes apart (leading offset),
  // groups of 8 key rows 1024 bytes apart; a K-step of 16 keys advances the start by 2048 bytes
  auto values = [&](int s, uint32_t slot, int half, bool first) {
    const uint32_t v_lo = v_lo0 + slot * (C::kTileBytes >> 4);
    tc_fence_after();
#pragma unroll
    for (int kk = 0; kk < kCols / 32; ++kk) {
      const int ks = half * (kCols / 32) + kk;
      if (leader)
        mma_ts(tmem + kTmemO + s * D, tmem + kTmemS + s * kCols + ks * 8, desc_from_lo(v_lo + ((ks * 2048) >> 4)), idesc_pv,
               (first && ks == 0) ? 0u : 1u);
    }
  };
#define NEED(bar, parity) if (!WAIT_ALL(bar, parity)) { ok = false; break; }
  for (int w = blockIdx.x; ok && w < p.total_work; w += gridDim.x, ++n_item) {
    if (n_item == 0) {                           // later items' first scores follow the previous item's last P V
      for (int s = 0; s < 2; ++s) {
        NEED(&sm.q_full[s], 0)
        if (s == 0) { NEED(&sm.kv_full[0], 0) }
        scores(s, 0);
        if (n_tiles == 1 && leader) mma_commit(&sm.q_empty[s]);
      }
      if (!ok) break;
      if (leader) mma_commit(&sm.kv_empty[0]);
    }
    const bool more_items = w + (int)gridDim.x < p.total_work;
    for (int t = 0; ok && t < n_tiles; ++t, ++g, m += 2) {
      const uint32_t v_slot = (m + 1) % kSlots, k_slot = (m + 2) % kSlots;
      const bool last = t == n_tiles - 1, next = !last || more_items;
      for (int s = 0; s < 2; ++s) {
        if (s == 0) { NEED(&sm.kv_full[v_slot], ((m + 1) / kSlots) & 1) }
        // the first P V of a work item overwrites O: the previous item's epilogue must have read it
        if (t == 0 && n_item > 0) { NEED(&sm.o_free[s], (n_item - 1) & 1) }
        NEED(&sm.p_full[s][0], g & 1)
        values(s, v_slot, 0, t == 0);
        // what the next scores need is looked at while the second half of P is on its way
        if (next) {
          if (s == 0) { NEED(&sm.kv_full[k_slot], ((m + 2) / kSlots) & 1) }
          if (last) { NEED(&sm.q_full[s], (n_item + 1) & 1) }
        }
        NEED(&sm.p_full[s][1], g & 1)
        values(s, v_slot, 1, false);
        if (leader) {
          if (last) mma_commit(&sm.o_full[s]);
          // (test hook: a withheld completion signal makes the bounded waits on it run out)
          if (s == 1 && (int)g != p.withhold_tile) mma_commit(&sm.kv_empty[v_slot]);
        }
        // (the scores overwrite P behind a P V that has been issued, not completed: MMAs of one thread are assumed to run in
        //  the order of issue, also where shape and accumulator differ)
        if (next) scores(s, k_slot);
        if (leader) {
          // Q is free behind the last scores that read it (of this item, or of a next item with one tile)
          if (next && (last ? n_tiles == 1 : t + 1 == n_tiles - 1)) mma_commit(&sm.q_empty[s]);
          if (s == 1 && next) mma_commit(&sm.kv_empty[k_slot]);
        }
      }
    }
  }
#undef NEED
  if (!ok && leader) flag_abort(sm, p, 300);
  __syncwarp();
  if (sm.abort_flag) {
    // TMEM must not be released while MMAs are still writing to it: wait (bounded) behind everything issued
    if (leader) mma_commit(&sm.mma_drain);
    int never = 0;
    mbar_wait_inline(&sm.mma_drain, 0, &never, p.wait_limit);
  }
}

template <int D>
__device__ void softmax_role(Shared& sm, const Params& p, uint32_t tmem, int s, int warp_in_group, int lane) {
  constexpr int kHalf = kCols / 2;
  const unsigned full = 0xffffffffu;
  const uint32_t lane_base = tmem + ((uint32_t)(warp_in_group * 32) << 16);
  const uint32_t t_s = lane_base + kTmemS + s * kCols, t_o = lane_base + kTmemO + s * D;
  const int row = warp_in_group * 32 + lane;
  const int n_tiles = ceil_div(p.N, kCols);
  const float sl2 = p.scale * 1.4426950408889634f;
  uint32_t g = 0, n_item = 0;
  bool ok = true;
  for (int w = blockIdx.x; ok && w < p.total_work; w += gridDim.x, ++n_item) {
    float m_used = -INFINITY, l = 0.f;
    for (int t = 0; t < n_tiles; ++t, ++g) {
      const int cols_valid = p.N - t * kCols;
      if (!WAIT_ALL(&sm.s_full[s], g & 1)) { ok = false; break; }
      tc_fence_after();
      uint32_t sr[kCols];
      auto half_max = [&](int c0) {
        constexpr int kQ = kHalf / 4;
        float m[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) m[x] = -INFINITY;
#pragma unroll
        for (int c = 0; c < kQ; c += 2)
#pragma unroll
          for (int x = 0; x < 4; ++x)
            m[x] = fmaxf(fmaxf(m[x], __uint_as_float(sr[c0 + x * kQ + c])), __uint_as_float(sr[c0 + x * kQ + c + 1]));
        return fmaxf(fmaxf(m[0], m[1]), fmaxf(m[2], m[3]));
      };
      auto mask_half = [&](int c0) {             // columns past the last token
#pragma unroll
        for (int c = 0; c < kHalf; ++c)
          if (c0 + c >= cols_valid) sr[c0 + c] = __float_as_uint(-INFINITY);
      };
      // the maximum of the first half is taken while the second half is on its way
      tmem_ld_cols<kHalf>(t_s, sr);
      tmem_ld_wait();
      tmem_ld_cols<kHalf>(t_s + kHalf, sr + kHalf);
      if (cols_valid < kCols) mask_half(0);
      float mx = half_max(0);
      tmem_ld_wait();
      if (cols_valid < kCols) mask_half(kHalf);
      mx = fmaxf(mx, half_max(kHalf)) * sl2;
      if (t == 0) {
        m_used = mx;
      } else if (__any_sync(full, mx > m_used + kRescaleThreshold)) {
        const float m_new = fmaxf(m_used, mx);
        const float f = (m_new == -INFINITY) ? 1.f : ex2(m_used - m_new);
        // (P V of the previous tile has landed in O: it was issued before the scores of this one)
#pragma unroll 1
        for (int c = 0; c < D / 16; ++c) {
          uint32_t o[16];
          tmem_ld_32x32b_x16(t_o + c * 16, o);
          tmem_ld_wait();
#pragma unroll
          for (int x = 0; x < 16; ++x) o[x] = __float_as_uint(__uint_as_float(o[x]) * f);
          tmem_st_32x32b_x16(t_o + c * 16, o);
        }
        l *= f;
        m_used = m_new;
      }
      // P = exp2(sl2 S - m), scaled as packed fp32 pairs.  The row sum is that of the rounded P, the weights that P V
      // uses: with one maximum per row the sum of the unrounded P has a larger error against 64 bits (12 heads,
      // 11 160 tokens with sink tokens, d = 128: 1.93e-3; so 1.83e-3; fwd_sm100.cu with a maximum per column half
      // 1.90e-3).
      const float nm = (m_used == -INFINITY) ? 0.f : -m_used;   // a row without a finite logit yet: all P = 0
      const float2 sl2_2 = make_float2(sl2, sl2), nm2 = make_float2(nm, nm);
      float2 s_a = make_float2(0.f, 0.f), s_b = make_float2(0.f, 0.f);
      auto exps = [&](int c0, int n) {           // columns [c0, c0 + n), bf16 pairs to sr[c0 / 2 ...]
#pragma unroll
        for (int c = 0; c < n; c += 4) {
          const uint32_t* x = sr + c0 + c;
          const float2 xa = __ffma2_rn(make_float2(__uint_as_float(x[0]), __uint_as_float(x[1])), sl2_2, nm2);
          const float2 xb = __ffma2_rn(make_float2(__uint_as_float(x[2]), __uint_as_float(x[3])), sl2_2, nm2);
          const float2 ea = make_float2(ex2(xa.x), ex2(xa.y));
          const float2 eb = make_float2(ex2(xb.x), ex2(xb.y));
          __nv_bfloat162 lo = __floats2bfloat162_rn(ea.x, ea.y);
          __nv_bfloat162 hi = __floats2bfloat162_rn(eb.x, eb.y);
          sr[(c0 + c) / 2] = *reinterpret_cast<uint32_t*>(&lo);
          sr[(c0 + c) / 2 + 1] = *reinterpret_cast<uint32_t*>(&hi);
          s_a = add_bf16x2(s_a, sr[(c0 + c) / 2]);
          s_b = add_bf16x2(s_b, sr[(c0 + c) / 2 + 1]);
        }
      };
      auto arrive = [&](int half) {
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.p_full[s][half]);
      };
      exps(0, kHalf);
      tmem_st_32x32b_x32(t_s, *reinterpret_cast<uint32_t(*)[32]>(&sr[0]));
      // the store of the first half completes behind the first exponentials of the second
      exps(kHalf, kHalf / 4);
      arrive(0);
      exps(kHalf + kHalf / 4, 3 * kHalf / 4);
      tmem_st_32x32b_x32(t_s + 32, *reinterpret_cast<uint32_t(*)[32]>(&sr[32]));
      arrive(1);
      const float2 sum = __fadd2_rn(s_a, s_b);
      l += sum.x + sum.y;
    }
    if (!ok) break;
    // ---- O / l
    const Item it = item_at(p, w);
    const int q_row = it.row + s * kRowsQ + row;
    __nv_bfloat16* orow = p.out + (size_t)it.b * (size_t)p.st.batch + (size_t)it.h * (size_t)p.st.head +
                          (size_t)q_row * (size_t)p.st.row;
    if (!WAIT_ALL(&sm.o_full[s], n_item & 1)) { ok = false; break; }
    tc_fence_after();
    const bool mass = m_used != -INFINITY;       // a row without any finite logit is zero
    const float inv = 1.f / l;
#pragma unroll 1
    for (int c = 0; c < D / 32; ++c) {
      uint32_t a[32];
      tmem_ld_32x32b_x32(t_o + c * 32, a);
      tmem_ld_wait();
      if (c == D / 32 - 1) {                     // the accumulator is in registers: it may be overwritten
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&sm.o_free[s]);
      }
      if (q_row < p.N) {
#pragma unroll
        for (int x = 0; x < 2; ++x) {            // 32 bytes (16 channels) per store
          uint32_t pw[8];
#pragma unroll
          for (int y = 0; y < 8; ++y) {
            const int e0 = x * 16 + 2 * y;
            __nv_bfloat162 hh = __floats2bfloat162_rn(mass ? __uint_as_float(a[e0]) * inv : 0.f,
                                                      mass ? __uint_as_float(a[e0 + 1]) * inv : 0.f);
            pw[y] = *reinterpret_cast<uint32_t*>(&hh);
          }
          if (p.out_aligned32) {
            st_global_v8(orow + c * 32 + x * 16, pw);
          } else {                               // the interface only asks for 16-byte alignment
            uint4* dst = reinterpret_cast<uint4*>(orow + c * 32 + x * 16);
            dst[0] = make_uint4(pw[0], pw[1], pw[2], pw[3]);
            dst[1] = make_uint4(pw[4], pw[5], pw[6], pw[7]);
          }
        }
      }
    }
  }
  if (!ok) flag_abort(sm, p, 400);
}

// counts = Nk and the debug mask's bits = 1 for the query blocks of this CTA's work items
__device__ void counts_role(const Params& p, int block, int lane) {
  const int words = ceil_div(p.Nk, 32), per = 2 * kRowsQ / block;
  for (int w = blockIdx.x; w < p.total_work; w += gridDim.x) {
    const int bh = w / p.items_per_head, i0 = (w - bh * p.items_per_head) * per;
    for (int x = 0; x < per && i0 + x < p.Nq; ++x) {
      const size_t r = (size_t)bh * p.Nq + i0 + x;
      if (p.counts && lane == 0) p.counts[r] = p.Nk;
      if (p.mask_out)
        for (int y = lane; y < words; y += 32)
          p.mask_out[r * words + y] = y == words - 1 && p.Nk % 32 ? (1u << (p.Nk % 32)) - 1u : 0xffffffffu;
    }
  }
}

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
fwd_sm100_dense_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                       const __grid_constant__ CUtensorMap tm_v, const Params p, int block) {
  using C = Cfg<D>;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* sQ = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* sKV = sQ + 2 * C::kTileBytes;
  Shared& sm = *reinterpret_cast<Shared*>(sKV + kSlots * C::kTileBytes);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    sm.abort_flag = 0;
    for (int i = 0; i < kSlots; ++i) { mbar_init(&sm.kv_full[i], 1); mbar_init(&sm.kv_empty[i], 1); }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sm.q_full[s], 1); mbar_init(&sm.q_empty[s], 1);
      mbar_init(&sm.s_full[s], 1);
      mbar_init(&sm.p_full[s][0], 4); mbar_init(&sm.p_full[s][1], 4);
      mbar_init(&sm.o_full[s], 1); mbar_init(&sm.o_free[s], 4);
    }
    mbar_init(&sm.mma_drain, 1);
    fence_mbar_init();
  }
  if (warp == kWarpProducer && lane == 0) { prefetch_tensormap(&tm_q); prefetch_tensormap(&tm_k); prefetch_tensormap(&tm_v); }
  if (warp == 0) { tmem_alloc(&sm.tmem_base, kTmemCols); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_base;
  kernel_wait();

  // A softmax thread holds a whole row of scores: it takes registers over from the other roles.
  if (warp < 8) {
    set_max_registers_up<kRegsSoftmax>();
    softmax_role<D>(sm, p, tmem, warp / 4, warp % 4, lane);
  } else {
    set_max_registers_down<kRegsOther>();
    if (warp == kWarpMma) mma_role<D>(sm, p, sQ, sKV, tmem);
    else if (warp == kWarpProducer && lane == 0) producer_role<D>(sm, p, sQ, sKV, &tm_q, &tm_k, &tm_v);
    else if (warp == kWarpCounts) counts_role(p, block, lane);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

template <int D>
cudaError_t launch_instance(const Problem& p, const Maps& m, const Params& prm, int grid, cudaStream_t stream) {
  // the roles share out what the launch brings, which is the compiler's choice within the launch bounds
  static std::atomic<bool> enough{false};
  if (!enough) {
    cudaFuncAttributes a{};
    const cudaError_t e = cudaFuncGetAttributes(&a, fwd_sm100_dense_kernel<D>);
    if (e != cudaSuccess) return e;
    if (a.numRegs < kRegsLaunch) return cudaErrorInvalidConfiguration;
    enough = true;
  }
  const size_t smem = 1024 + (2 + kSlots) * Cfg<D>::kTileBytes + sizeof(Shared);
  return launch_after(fwd_sm100_dense_kernel<D>, dim3(grid), kThreads, smem, smem, 0, stream, m.q, m.k, m.v, prm, p.block_q);
}

}  // namespace

cudaError_t launch_dense(const Problem& p, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                         __nv_bfloat16* out, const WsPtrs& ws, int32_t* counts, uint32_t* mask_out, int sms,
                         long long wait_limit, int withhold_tile, cudaStream_t stream, int* n_launches) {
  Maps m;
  Params prm;
  if (!prepare(p, q, k, v, out, ws, nullptr, counts, mask_out, kCols, &m, &prm)) return cudaErrorInvalidValue;
  prm.wait_limit = wait_limit;
  prm.withhold_tile = withhold_tile;
  prm.items_per_head = ceil_div(p.N, 2 * kRowsQ);
  prm.total_work = p.BH * prm.items_per_head;
  const int grid = prm.total_work < sms ? prm.total_work : sms;
  if (n_launches) *n_launches += 1;
  return p.d == 128 ? launch_instance<128>(p, m, prm, grid, stream) : launch_instance<64>(p, m, prm, grid, stream);
}

}  // namespace fwd
}  // namespace sol
