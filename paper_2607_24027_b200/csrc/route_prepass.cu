// Optional routing pre-pass (SOL_ROUTING_PREPASS): the comparison of Eq. (4),
//   s_ij = scale * Qbar_i . KC_j  >  tau_i   (strict),
// evaluated for every (query block, key block) pair before the fused kernel runs, and kept as ONE
// BIT per pair in the caller's mask buffer.  The proxy scores themselves still never reach memory:
// they live in the tensor memory of this kernel for the length of one 128 x 128 tile.  The fused kernel's
// router then only turns the bits into tile records, which takes its shared-memory and
// instruction-issue load off the scheduler it shares with two softmax warps.
//
// Algorithm 1 routes inside the attention loop; this is the same decision taken earlier, so the
// default stays the in-kernel router and this path is an option for low routing densities.
#include "fwd_sm100_common.cuh"

namespace sol {
namespace {

using namespace ptx;

// The products are those of fp32 numbers: each is cut into three bf16 parts, x = x1 + x2 + x3 (8 significant bits each, so the
// sum is x), and of the nine products of parts the six that matter in fp32 are formed by the tensor core,
//   x y = x1 y1 + (x1 y2 + x2 y1 + x2 y2 + x1 y3 + x3 y1),   the rest 2^-24 of |x| |y| at the most, 2^-27 as a rule.
// Products of bf16 parts are exact in fp32.  The small terms have an accumulator of their own, so that they are not
// rounded at the size of the large ones, and the first term has two: the tensor core rounds towards zero when it adds, and
// every addition counts.  Error of the scores against 64 bits, relative 2-norm (packed FMAs of proxy_tile.cuh / this with one, two,
// three accumulators of the first term), d = 128: 40 x 591 x 591 blocks 1.44e-7 / - / 1.31e-7 / 1.11e-7, 24 x 32 x 32
// 1.53e-7 / 2.81e-7 / 1.35e-7 / 1.32e-7; d = 64, 16 x 175 x 175 1.06e-7 / 1.09e-7 / 0.72e-7 / 0.69e-7.
//
// What this cannot form is formed with FMAs instead, in the order in which proxy_tile.cuh forms it (`direct_score`):
//   - a tile with an infinity, a NaN or a number from 2^60 on.  The first two have no parts.  Where products leave the range of
//     fp32, parts of both signs make a NaN of what the FMAs make an infinity (x = y = 1.0039 * 2^64: x1 y1 = inf, x1 y2 = -inf),
//     and the tensor core, which adds 16 products before it rounds, may see no overflow at all;
//   - a tile with a number below 2^-50 that is not zero, whose parts' products can be too small for fp32 to hold;
//   - a tile whose MMAs did not retire within the wait limit.  So the bits are right in that case too, and this
//     kernel has no error to report.
//
// 40 heads x 591 x 591 blocks, d = 128: 113 us with packed FMAs on the CUDA cores, 35 us so (two accumulators; 128 x 64 tiles
// 49 us; 0.7 us for looking at the range of the numbers); 24 x 32 x 32 blocks 10.3 / 6.4 us.  Its floor is the tensor core's: 1000
// tiles of 48 MMAs, 13 us; the rest is cutting (a third of the instructions) and the comparison, which two CTAs per SM
// overlap with the other's MMAs in part.
constexpr int kTile = 128;                       // query blocks per CTA
constexpr int kKeys = 128;                       // key blocks per CTA
constexpr int kChunk = 64;                       // channels in shared memory at a time
constexpr int kPartBytes = kTile * kChunk * 2;   // one bf16 part of one operand: a 128-byte row per block, 128-byte swizzle
constexpr int kThreadsMask = 256;
constexpr int kKeyPartBytes = kKeys * kChunk * 2;
constexpr int kMains = 2;                        // accumulators of the first term
constexpr int kMaskCols = 512;                   // tensor-memory columns: kMains + 1 accumulators of kKeys, a power of two

struct MaskShared {                              // behind the parts
  uint64_t done;                                 // the MMAs of a chunk have retired
  uint64_t drain;                                // a wait for that ran out: all MMAs issued have retired
  uint32_t tmem;
};
constexpr size_t kMaskSmem = 3 * (kPartBytes + kKeyPartBytes) + sizeof(MaskShared);

struct Parts { uint2 p[3]; };                    // four channels: three parts of bf16

__device__ __forceinline__ Parts split(float4 v) {
  Parts r;
  const float x[4] = {v.x, v.y, v.z, v.w};
  float rest[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) rest[i] = x[i];
#pragma unroll
  for (int part = 0; part < 3; ++part) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(rest[0], rest[1]), hi = __floats2bfloat162_rn(rest[2], rest[3]);
    r.p[part] = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    rest[0] -= __uint_as_float(r.p[part].x << 16);
    rest[1] -= __uint_as_float(r.p[part].x & 0xffff0000u);
    rest[2] -= __uint_as_float(r.p[part].y << 16);
    rest[3] -= __uint_as_float(r.p[part].y & 0xffff0000u);
  }
  return r;
}
// Smallest and largest magnitude of the numbers seen so far, by their first parts (in 16-bit halves).  `least` is one less than
// that: zero less one is the largest number there is, so that zeros do not count.
struct Range {
  uint32_t least = 0xffffffffu, most = 0;
  __device__ __forceinline__ void add(uint2 parts) {
    const uint32_t a = parts.x & 0x7fff7fffu, b = parts.y & 0x7fff7fffu;
    least = __viaddmin_u16x2(b, 0xffffffffu, __viaddmin_u16x2(a, 0xffffffffu, least));
    most = __vimax3_u16x2(a, b, most);
  }
  __device__ __forceinline__ bool left() const {
    return min(least & 0xffffu, least >> 16) + 1 < (127 - 50) << 7 || max(most & 0xffffu, most >> 16) >= (127 + 60) << 7;
  }
};

__device__ __noinline__ float direct_score(const float* __restrict__ q, const float* __restrict__ k, int d) {
  float even = 0.f, odd = 0.f;
  for (int c = 0; c < d; c += 2) {
    even = fmaf(q[c], k[c], even);
    odd = fmaf(q[c + 1], k[c + 1], odd);
  }
  return even + odd;
}

// grid (ceil(Nk / 128), ceil(Nq / 128), BH).  mask[bh][i][w]: bit j % 32 of word j / 32 = block j routed.
__global__ void __launch_bounds__(kThreadsMask, 2)
mask_prepass_kernel(const float* __restrict__ qbar, const float* __restrict__ kc, const float* __restrict__ tau,
                    const uint8_t* __restrict__ forced, uint32_t* __restrict__ mask, int Nq, int Nk, int d, float scale,
                    long long wait_limit, int withhold) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* parts = smem_raw;
  MaskShared& sm = *reinterpret_cast<MaskShared*>(smem_raw + 3 * (kPartBytes + kKeyPartBytes));
  const int tid = threadIdx.x, warp = tid / 32, lane = tid % 32;
  const int bh = blockIdx.z, i0 = blockIdx.y * kTile, j0 = blockIdx.x * kKeys;
  if (tid == 0) { mbar_init(&sm.done, 1); mbar_init(&sm.drain, 1); fence_mbar_init(); }
  __syncthreads();
  kernel_wait();
  const float* q = qbar + ((size_t)bh * Nq + i0) * d;
  const float* k = kc + ((size_t)bh * Nk + j0) * d;
  const int nq = min(kTile, Nq - i0), nk = min(kKeys, Nk - j0);
  const uint32_t idesc = make_idesc_bf16(kTile, kKeys, false, false);
  const uint32_t lo0 = (smem_addr(parts) >> 4) | (1u << 16);
  const bool leader = warp == 0 && elect_one();  // issues all MMAs and their completion signals
  int never = 0;
  uint32_t tmem = 0;
  Range range;
  bool ok = true;                                // no wait has run out
  for (int c0 = 0, chunk = 0; c0 < d; c0 += kChunk, ++chunk) {
    // 16 threads per row, 16 rows at a time: query blocks, then key blocks
    const int c4 = tid % 16;
    constexpr int kQ = kTile / 16, kK = kKeys / 16;
    float4 v[kQ + kK];
#pragma unroll
    for (int x = 0; x < kQ + kK; ++x) {
      const int r = tid / 16 + 16 * (x < kQ ? x : x - kQ);
      v[x] = r < (x < kQ ? nq : nk) ? __ldg(reinterpret_cast<const float4*>((x < kQ ? q : k) + (size_t)r * d + c0) + c4)
                                    : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    if (chunk > 0) ok = mbar_wait(&sm.done, (chunk - 1) & 1, &never, wait_limit);   // the parts of the chunk before have been read
#pragma unroll
    for (int x = 0; x < kQ + kK; ++x) {
      const int r = tid / 16 + 16 * (x < kQ ? x : x - kQ);     // below 128 or kKeys: the row stays inside its part
      const Parts s = split(v[x]);
      range.add(s.p[0]);
      unsigned char* dst = parts + (x < kQ ? 0 : 3 * kPartBytes) + r * 128 + (((c4 / 2) ^ (r & 7)) * 16) + (c4 & 1) * 8;
#pragma unroll
      for (int part = 0; part < 3; ++part) *reinterpret_cast<uint2*>(dst + part * (x < kQ ? kPartBytes : kKeyPartBytes)) = s.p[part];
    }
    fence_proxy_async_smem();
    if (chunk == 0) {
      // this late, so that of two CTAs on an SM one loads and cuts while the other has the tensor memory
      if (warp == 0) { tmem_alloc(&sm.tmem, kMaskCols); tmem_relinquish(); }
      tc_fence_before();
    }
    ok = __syncthreads_and(ok);
    tmem = *const_cast<volatile uint32_t*>(&sm.tmem);
    if (!ok) break;                              // (a wait ran out: not in the first chunk)
    if (warp == 0) {
      tc_fence_after();
      constexpr int kP[6][2] = {{0, 1}, {1, 0}, {1, 1}, {0, 2}, {2, 0}, {0, 0}};   // the first term comes last
#pragma unroll
      for (int t = 0; t < 6; ++t)
#pragma unroll
        for (int ks = 0; ks < kChunk / 16; ++ks) {
          const uint32_t a = lo0 + ((kP[t][0] * kPartBytes + ks * 32) >> 4), b = lo0 + ((3 * kPartBytes + kP[t][1] * kKeyPartBytes + ks * 32) >> 4);
          const int acc = t == 5 ? ks % kMains : kMains;
          const bool fresh = chunk == 0 && (t == 5 ? ks < kMains : (t == 0 && ks == 0));
          if (leader) mma_ss(tmem + acc * kKeys, fwd::desc_from_lo(a), fwd::desc_from_lo(b), idesc, fresh ? 0u : 1u);
        }
      // (test hook: a withheld completion signal makes the waits on it run out)
      if (leader && chunk != withhold) mma_commit(&sm.done);
    }
    __syncwarp();
  }
  if (ok) ok = mbar_wait(&sm.done, (ceil_div(d, kChunk) - 1) & 1, &never, wait_limit);
  tc_fence_after();
  ok = __syncthreads_and(ok);
  const bool direct = __syncthreads_or(range.left() || !ok);
  // thread = query block, half of the key blocks each
  const int row = (warp % 4) * 32 + lane, col0 = (warp / 4) * (kKeys / 2);
  const int i = i0 + row, words = ceil_div(Nk, 32);
  const float t = i < Nq ? tau[(size_t)bh * Nq + i] : 0.f;
#pragma unroll
  for (int c = 0; c < kKeys / 64; ++c) {
    const int j = j0 + col0 + 32 * c;            // this word's first key block
    uint32_t word = 0;
    if (!direct) {
      uint32_t acc[kMains + 1][32];
#pragma unroll
      for (int x = 0; x <= kMains; ++x)
        tmem_ld_32x32b_x32(tmem + ((uint32_t)((warp % 4) * 32) << 16) + x * kKeys + col0 + 32 * c, acc[x]);
      tmem_ld_wait();
#pragma unroll
      for (int b = 0; b < 32; ++b) {
        float dot = __uint_as_float(acc[0][b]);
#pragma unroll
        for (int x = 1; x <= kMains; ++x) dot += __uint_as_float(acc[x][b]);
        word |= (scale * dot > t ? 1u : 0u) << b;
      }
    } else if (row < nq) {
      for (int b = 0; b < 32 && j + b < Nk; ++b) {
        const float dot = direct_score(q + (size_t)row * d, k + (size_t)(j - j0 + b) * d, d);
        word |= (scale * dot > t ? 1u : 0u) << b;
      }
    }
    __syncwarp();
    word |= __ballot_sync(0xffffffffu, forced && j + lane < Nk && forced[j + lane]);
    if (j + 32 > Nk) word &= j < Nk ? (1u << (Nk - j)) - 1u : 0u;
    if (i < Nq && j < Nk) mask[((size_t)bh * Nq + i) * words + j / 32] = word;
  }
  if (warp == 0 && !ok) {
    // the tensor memory must not be released while MMAs still write to it: wait (bounded) behind all that were issued
    if (leader) mma_commit(&sm.drain);
    mbar_wait(&sm.drain, 0, &never, wait_limit);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, kMaskCols);
}

}  // namespace

cudaError_t launch_route_prepass(const Problem& p, const WsPtrs& ws, const float* tau, uint32_t* mask,
                                 cudaStream_t stream, int* n_launches) {
  const dim3 grid(ceil_div(p.Nk, kKeys), ceil_div(p.Nq, kTile), p.BH);
  if (n_launches) *n_launches += 1;
  return launch_after(mask_prepass_kernel, grid, kThreadsMask, kMaskSmem, kMaskSmem, 0, stream, ws.qbar, ws.kc, tau, p.forced,
                      mask, p.Nq, p.Nk, p.d, p.scale, fwd::g_wait_limit, fwd::g_withhold_tile);
}

}  // namespace sol
