// fp32 product of pooled queries and pooled keys, one 128 x 64 tile per CTA, left in registers: what the materialised
// baselines write out as the proxy map.  (The routing pre-pass forms its products on the tensor core, route_prepass.cu.)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace sol {

// 256 threads; thread (ty, tx) = (tid / 16, tid % 16) owns rows ty + 16 a (a < 8) and columns tx + 16 b (b < 4).
// FMA-bound: every 16-byte read of a row feeds four packed FMAs per row of the other side, 12 reads per 64 FMAs
// (a 4 x 4 patch with scalar reads needs 8 per 16, and runs at shared-memory speed).  Chunks of 32 channels are
// copied asynchronously, two deep.  The packed pairs run over the channels, so an accumulator is the sum of its even
// and its odd channels.
constexpr int kProxyRows = 128, kProxyCols = 64;
constexpr int kProxyChunk = 32, kProxyLd = kProxyChunk + 4;   // rows 4 banks apart: no bank conflicts
constexpr size_t kProxySmem = 2 * sizeof(float) * (kProxyRows + kProxyCols) * kProxyLd;

// kAligned: q and k are 16-byte aligned.  d is a multiple of 32.  Rows past nq / nk count as zero.
template <bool kAligned>
__device__ __forceinline__ void proxy_tile(const float* __restrict__ q, const float* __restrict__ k, int nq, int nk, int d,
                                           float* smem, float (&dot)[8][4]) {
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  auto load = [&](int c0, float* buf) {
#pragma unroll
    for (int x = 0; x < (kProxyRows + kProxyCols) * (kProxyChunk / 4) / 256; ++x) {
      const int e = tid + 256 * x, r = e / (kProxyChunk / 4), c = (e % (kProxyChunk / 4)) * 4;
      const bool is_q = r < kProxyRows;
      const int row = is_q ? r : r - kProxyRows;
      const bool ok = row < (is_q ? nq : nk);
      const float* src = (is_q ? q : k) + (ok ? (size_t)row * d + c0 + c : 0);
      float* dst = buf + r * kProxyLd + c;
      if constexpr (kAligned) {
        const uint32_t s = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
        const int bytes = ok ? 16 : 0;                        // the rest is filled with zeros
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s), "l"(src), "r"(bytes) : "memory");
      } else {
#pragma unroll
        for (int y = 0; y < 4; ++y) dst[y] = ok ? src[y] : 0.f;
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  constexpr int kBuf = (kProxyRows + kProxyCols) * kProxyLd;
  float2 acc[8][4];
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = make_float2(0.f, 0.f);
  load(0, smem);
  for (int c0 = 0, n = 0; c0 < d; c0 += kProxyChunk, ++n) {
    if (c0 + kProxyChunk < d) load(c0 + kProxyChunk, smem + ((n + 1) & 1) * kBuf);
    else asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    const float* qs = smem + (n & 1) * kBuf + ty * kProxyLd;
    const float* ks = smem + (n & 1) * kBuf + (kProxyRows + tx) * kProxyLd;
#pragma unroll 2
    for (int c = 0; c < kProxyChunk; c += 4) {
      float4 kv[4];
#pragma unroll
      for (int b = 0; b < 4; ++b) kv[b] = *reinterpret_cast<const float4*>(ks + 16 * b * kProxyLd + c);
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        const float4 qv = *reinterpret_cast<const float4*>(qs + 16 * a * kProxyLd + c);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          acc[a][b] = __ffma2_rn(make_float2(qv.x, qv.y), make_float2(kv[b].x, kv[b].y), acc[a][b]);
          acc[a][b] = __ffma2_rn(make_float2(qv.z, qv.w), make_float2(kv[b].z, kv[b].w), acc[a][b]);
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) dot[a][b] = acc[a][b].x + acc[a][b].y;
}

}  // namespace sol
