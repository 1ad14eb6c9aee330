// sol_attn_route_materialized: the two routing baselines the paper measures its on-the-fly
// thresholding against (introduction, limitation L1; routing-latency figure): the block proxy map
// s_ij = scale * Qbar_i . KC_j (Eq. 3) is WRITTEN TO MEMORY, every row is sorted, and
//   top-k keeps the k highest-scoring key blocks of each query block,
//   top-p keeps blocks in descending order until their share of the row's softmax mass reaches p.
// The result is handed back as routing indices, counts and an equivalent per-row cutoff tau (the
// midpoint between the last kept and the first dropped score), which the fused kernel accepts as
// its threshold array -- so both policies can also drive the single-pass kernel.
#include <math.h>

#include "common.cuh"
#include "proxy_tile.cuh"

namespace {

constexpr int kMaxRow = 8192;          // longest proxy row the in-shared-memory sort takes

// map[bh][i][j] = scale * sum_c qbar[bh][i][c] * kc[bh][j][c]; grid (ceil(Nk/64), ceil(Nq/128), BH).
// 40 heads x 256 x 256 blocks, d = 128: 27 us (38 us with scalar shared-memory reads).
template <bool kAligned>
__global__ void __launch_bounds__(256, 2) proxy_map_kernel(const float* __restrict__ qbar, const float* __restrict__ kc,
                                                           float* __restrict__ map, int Nq, int Nk, int d, float scale) {
  extern __shared__ __align__(16) float smem_f[];
  const int bh = blockIdx.z, i0 = blockIdx.y * sol::kProxyRows, j0 = blockIdx.x * sol::kProxyCols;
  const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
  float dot[8][4];
  sol::proxy_tile<kAligned>(qbar + ((size_t)bh * Nq + i0) * d, kc + ((size_t)bh * Nk + j0) * d, Nq - i0, Nk - j0, d,
                            smem_f, dot);
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const int i = i0 + ty + 16 * a;
    if (i >= Nq) continue;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int j = j0 + tx + 16 * b;
      if (j < Nk) map[((size_t)bh * Nq + i) * Nk + j] = scale * dot[a][b];
    }
  }
}

// true when (va, ia) sorts before (vb, ib): higher score first, lower block index on ties
__device__ __forceinline__ bool before(float va, int ia, float vb, int ib) {
  return va > vb || (va == vb && ia < ib);
}

// One warp per proxy row of up to 1024 scores: the row is sorted in registers, lane l holding places
// [l kPer, (l + 1) kPer).  An entry is one 64-bit key that sorts descending as wanted: the score in an unsigned form
// of the same order, then the complement of the block index (lower index first on ties; -0 is made +0, so that the two
// tie as they compare).  Steps of the bitonic network inside a lane are register moves, the others one shuffle each;
// 40 heads x 256 rows x 256 scores: 27 us, where a CTA per row with the keys in shared memory and a barrier
// after each of 36 steps took 100 us.  Longer rows would spill; they keep that kernel (below).
__device__ __forceinline__ uint64_t sort_key(float v, int j) {
  const uint32_t x = __float_as_uint(v + 0.f);
  const uint32_t o = (x & 0x80000000u) ? ~x : x | 0x80000000u;
  return (uint64_t)o << 32 | (uint32_t)~j;
}
__device__ __forceinline__ float key_score(uint64_t k) {
  const uint32_t o = (uint32_t)(k >> 32);
  return __uint_as_float((o & 0x80000000u) ? o & 0x7fffffffu : ~o);
}

constexpr int kSelectWarps = 4;

template <int kPer>
__global__ void __launch_bounds__(32 * kSelectWarps)
row_select_warp_kernel(const float* __restrict__ map, long long n_rows, int Nk, int policy, float param,
                       int32_t* __restrict__ order, float* __restrict__ tau, int32_t* __restrict__ counts) {
  __shared__ float val[kSelectWarps][32 * kPer];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const long long row = (long long)blockIdx.x * kSelectWarps + warp;
  if (row >= n_rows) return;                     // whole warps leave; there is no block-wide barrier
  const float* src = map + row * Nk;
  uint64_t key[kPer];
#pragma unroll
  for (int r = 0; r < kPer; ++r) {               // coalesced: any start order will do
    const int j = r * 32 + lane;
    key[r] = j < Nk ? sort_key(src[j], j) : 0;   // 0 sorts behind every score
  }
#pragma unroll
  for (int size = 2; size <= 32 * kPer; size <<= 1) {
#pragma unroll
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      if (stride >= kPer) {                      // partner in another lane
        const int lane_stride = stride / kPer;
        const bool lower = (lane & lane_stride) == 0;
        const bool descending = ((lane * kPer) & size) == 0;
#pragma unroll
        for (int r = 0; r < kPer; ++r) {
          const uint64_t other = __shfl_xor_sync(0xffffffffu, key[r], lane_stride);
          const bool keep_max = lower == descending;
          key[r] = (key[r] > other) == keep_max ? key[r] : other;
        }
      } else {
#pragma unroll
        for (int r = 0; r < kPer; ++r) {
          if (r & stride) continue;
          const bool descending = size >= kPer ? ((lane * kPer) & size) == 0 : (r & size) == 0;
          const uint64_t a = key[r], b = key[r + stride];
          const bool swap = (a < b) == descending;
          key[r] = swap ? b : a;
          key[r + stride] = swap ? a : b;
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < kPer; ++r) val[warp][lane * kPer + r] = key_score(key[r]);
  __syncwarp();
  int c;
  if (policy == SOL_ROUTE_TOPK) {
    c = min(max((int)param, 0), Nk);
  } else {
    // share of the row's softmax mass held by the first c blocks; double so that the running sum
    // is not what decides a close call
    const int j0 = lane * kPer;
    const float top = val[warp][0];
    double local = 0.0;
    for (int j = j0; j < min(j0 + kPer, Nk); ++j) local += exp((double)val[warp][j] - (double)top);
    double run = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double x = __shfl_up_sync(0xffffffffu, run, o);
      if (lane >= o) run += x;
    }
    // (the total of the last lane with any mass: the lanes behind it add nothing, but in another order)
    const unsigned live = __ballot_sync(0xffffffffu, local != 0.0);
    const double total = __shfl_sync(0xffffffffu, run, live ? 31 - __clz(live) : 0);
    double before_lane = __shfl_up_sync(0xffffffffu, run, 1);
    if (lane == 0) before_lane = 0.0;
    const double need = (double)param * total;
    // the first c with mass(c) >= need; mass(c) = sum of the first c blocks.  The scan says in which lane that is; the
    // lane's own running sum may end a rounding below the scan's, and then its last block with any mass is the one.
    int first = Nk;
    if (before_lane < need && need <= run) {
      double mass = before_lane;
      for (int j = j0; j < min(j0 + kPer, Nk); ++j) {
        const double x = exp((double)val[warp][j] - (double)top);
        mass += x;
        if (x != 0.0) first = j + 1;
        if (mass >= need) break;
      }
    }
    c = __reduce_min_sync(0xffffffffu, first);
    if (need <= 0.0) c = 0;
  }
  if (order) {
    // through shared memory, so that the row is written in whole segments
    const float t_kept = c > 0 ? val[warp][c - 1] : 0.f, t_drop = c < Nk ? val[warp][c] : 0.f;
    __syncwarp();
    int* place = reinterpret_cast<int*>(val[warp]);
#pragma unroll
    for (int r = 0; r < kPer; ++r) place[lane * kPer + r] = (int)~(uint32_t)key[r];
    __syncwarp();
    for (int j = lane; j < Nk; j += 32) order[row * Nk + j] = place[j];
    if (lane == 0) tau[row] = c <= 0 ? INFINITY : (c >= Nk ? -INFINITY : 0.5f * (t_kept + t_drop));
  } else if (lane == 0) {
    tau[row] = c <= 0 ? INFINITY : (c >= Nk ? -INFINITY : 0.5f * (val[warp][c - 1] + val[warp][c]));
  }
  if (lane == 0 && counts) counts[row] = c;
}

// One CTA per proxy row: read it back from memory, sort it, apply the policy.
__global__ void __launch_bounds__(256) row_select_kernel(const float* __restrict__ map, int Nq, int Nk, int npad,
                                                         int policy, float param, int32_t* __restrict__ order,
                                                         float* __restrict__ tau, int32_t* __restrict__ counts) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* val = reinterpret_cast<float*>(smem_raw);
  int* idx = reinterpret_cast<int*>(val + npad);
  __shared__ double part[256];
  __shared__ double total_s;
  __shared__ int cut;
  const int i = blockIdx.x, bh = blockIdx.y;
  const size_t row = (size_t)bh * Nq + i;
  const float* src = map + row * Nk;
  for (int j = threadIdx.x; j < npad; j += 256) {
    val[j] = j < Nk ? src[j] : -INFINITY;
    idx[j] = j < Nk ? j : 0x7fffffff;
  }
  __syncthreads();
  // bitonic sort, descending
  for (int size = 2; size <= npad; size <<= 1) {
    for (int stride = size >> 1; stride > 0; stride >>= 1) {
      for (int t = threadIdx.x; t < npad / 2; t += 256) {
        const int lo = 2 * t - (t & (stride - 1));
        const int hi = lo + stride;
        const bool descending = (lo & size) == 0;
        const float va = val[lo], vb = val[hi];
        const int ia = idx[lo], ib = idx[hi];
        if (before(vb, ib, va, ia) == descending) {
          val[lo] = vb; val[hi] = va;
          idx[lo] = ib; idx[hi] = ia;
        }
      }
      __syncthreads();
    }
  }
  int c;
  if (policy == SOL_ROUTE_TOPK) {
    c = min(max((int)param, 0), Nk);
  } else {
    // share of the row's softmax mass held by the first c blocks; double so that the running sum
    // is not what decides a close call
    const int per = (npad + 255) / 256;
    const int j0 = threadIdx.x * per, j1 = min(j0 + per, Nk);
    const float top = val[0];
    double local = 0.0;
    for (int j = j0; j < j1; ++j) local += exp((double)val[j] - (double)top);
    part[threadIdx.x] = local;
    if (threadIdx.x == 0) cut = Nk;
    __syncthreads();
    if (threadIdx.x == 0) {
      double run = 0.0;
      for (int t = 0; t < 256; ++t) { const double x = part[t]; part[t] = run; run += x; }   // exclusive scan
      total_s = run;
    }
    __syncthreads();
    const double need = (double)param * total_s;
    double run = part[threadIdx.x];
    int first = Nk;
    // the first c with mass(c) >= need; mass(c) = sum of the first c blocks.  The scan says whose block that is; the
    // thread's own running sum may end a rounding below the scan's, and then its last block with any mass is the one.
    if (run < need && need <= run + local) {
      for (int j = j0; j < j1; ++j) {
        const double x = exp((double)val[j] - (double)top);
        run += x;
        if (x != 0.0) first = j + 1;
        if (run >= need) break;
      }
    }
    if (first < Nk) atomicMin(&cut, first);
    __syncthreads();
    c = cut;
    if (need <= 0.0) c = 0;
  }
  if (order)
    for (int j = threadIdx.x; j < Nk; j += 256) order[row * Nk + j] = idx[j];
  if (threadIdx.x == 0) {
    float t;
    if (c <= 0) t = INFINITY;
    else if (c >= Nk) t = -INFINITY;
    else t = 0.5f * (val[c - 1] + val[c]);
    tau[row] = t;
    if (counts) counts[row] = c;
  }
}

}  // namespace

extern "C" sol_status_t sol_attn_route_materialized(const float* qbar, const float* kc, int B, int H, int Nq, int Nk,
                                                    int d, float scale, int policy, float param, float* proxy_map,
                                                    int32_t* order, float* tau, int32_t* counts, sol_stream_t stream) {
  if (!qbar || !kc || !proxy_map || !tau) return SOL_ERR_INVALID_ARG;
  if (B <= 0 || H <= 0 || Nq <= 0 || Nk <= 0 || d <= 0 || param != param) return SOL_ERR_INVALID_ARG;
  if (policy != SOL_ROUTE_TOPK && policy != SOL_ROUTE_TOPP) return SOL_ERR_INVALID_ARG;
  if (policy == SOL_ROUTE_TOPP && (param < 0.f || param > 1.f)) return SOL_ERR_INVALID_ARG;
  if (d % 32 != 0 || Nk > kMaxRow || Nq > 65535 * 64 || (long long)B * H > 65535) return SOL_ERR_UNSUPPORTED_SHAPE;
  const int BH = B * H;
  const float sc = scale > 0.f ? scale : 1.0f / sqrtf((float)d);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const bool aligned = ((reinterpret_cast<uintptr_t>(qbar) | reinterpret_cast<uintptr_t>(kc)) & 15u) == 0;
  auto map_kernel = aligned ? proxy_map_kernel<true> : proxy_map_kernel<false>;
  if (cudaFuncSetAttribute(map_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sol::kProxySmem) != cudaSuccess)
    return SOL_ERR_CUDA;
  map_kernel<<<dim3((Nk + sol::kProxyCols - 1) / sol::kProxyCols, (Nq + sol::kProxyRows - 1) / sol::kProxyRows, BH), 256,
               sol::kProxySmem, st>>>(qbar, kc, proxy_map, Nq, Nk, d, sc);
  const long long n_rows = (long long)BH * Nq, n_cta = (n_rows + kSelectWarps - 1) / kSelectWarps;
  if (Nk <= 1024 && n_cta <= 0x7fffffffLL) {
    auto kernel = Nk <= 32 ? row_select_warp_kernel<1> : Nk <= 64 ? row_select_warp_kernel<2> : Nk <= 128 ? row_select_warp_kernel<4>
                  : Nk <= 256 ? row_select_warp_kernel<8> : Nk <= 512 ? row_select_warp_kernel<16> : row_select_warp_kernel<32>;
    kernel<<<(unsigned)n_cta, 32 * kSelectWarps, 0, st>>>(proxy_map, n_rows, Nk, policy, param, order, tau, counts);
  } else {
    int npad = 2;
    while (npad < Nk) npad <<= 1;
    const size_t smem = (size_t)npad * 8;
    // (the limit of the longest row, not of this call's: other threads may be launching the same kernel)
    if (cudaFuncSetAttribute(row_select_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxRow * 8) != cudaSuccess)
      return SOL_ERR_CUDA;
    row_select_kernel<<<dim3(Nq, BH), 256, smem, st>>>(proxy_map, Nq, Nk, npad, policy, param, order, tau, counts);
  }
  sol::count_launches(2);
  return cudaGetLastError() == cudaSuccess ? SOL_OK : SOL_ERR_CUDA;
}
