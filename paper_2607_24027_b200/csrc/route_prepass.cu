// Optional routing pre-pass (SOL_ROUTING_PREPASS): the comparison of Eq. (4),
//   s_ij = scale * Qbar_i . KC_j  >  tau_i   (strict),
// evaluated for every (query block, key block) pair before the fused kernel runs, and kept as ONE
// BIT per pair in the caller's mask buffer.  The proxy scores themselves still never reach memory:
// they live in the registers of this kernel for the length of one 128 x 64 tile.  The fused kernel's
// router then only turns the bits into tile records, which takes its shared-memory and
// instruction-issue load off the scheduler it shares with two softmax warps.
//
// Algorithm 1 routes inside the attention loop; this is the same decision taken earlier, so the
// default stays the in-kernel router and this path is an option for low routing densities.
#include "common.cuh"
#include "proxy_tile.cuh"

namespace sol {
namespace {

// grid (ceil(Nk / 64), ceil(Nq / 128), BH).  mask[bh][i][w]: bit j % 32 of word j / 32 = block j routed.
// 40 heads x 591 x 591 blocks, d = 128: 120 us (4.2 GFLOP with the padding of the tiles); 188 us with 4 x 4
// patches of a 64 x 64 tile and scalar shared-memory reads.
__global__ void __launch_bounds__(256, 2) mask_prepass_kernel(const float* __restrict__ qbar, const float* __restrict__ kc,
                                                              const float* __restrict__ tau,
                                                              const uint8_t* __restrict__ forced,
                                                              uint32_t* __restrict__ mask, int Nq, int Nk, int d,
                                                              float scale) {
  extern __shared__ __align__(16) float smem_f[];
  const int bh = blockIdx.z, i0 = blockIdx.y * kProxyRows, j0 = blockIdx.x * kProxyCols;
  const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
  float dot[8][4];
  kernel_wait();
  proxy_tile<true>(qbar + ((size_t)bh * Nq + i0) * d, kc + ((size_t)bh * Nk + j0) * d, Nq - i0, Nk - j0, d, smem_f, dot);
  bool force[4];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int j = j0 + tx + 16 * b;
    force[b] = forced && j < Nk && forced[j];
  }
  // a warp holds two rows (16 lanes each): two votes make a row's 32-bit word
  const int words = ceil_div(Nk, 32);
#pragma unroll
  for (int a = 0; a < 8; ++a) {
    const int i = i0 + ty + 16 * a;
    const float t = i < Nq ? tau[(size_t)bh * Nq + i] : 0.f;
    uint32_t vote[4];
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int j = j0 + tx + 16 * b;
      vote[b] = __ballot_sync(0xffffffffu, j < Nk && (scale * dot[a][b] > t || force[b]));
      if (threadIdx.x & 16) vote[b] >>= 16;
    }
    if (tx < 2 && i < Nq && j0 / 32 + tx < words)
      mask[((size_t)bh * Nq + i) * words + j0 / 32 + tx] =
          tx == 0 ? (vote[0] & 0xffffu) | vote[1] << 16 : (vote[2] & 0xffffu) | vote[3] << 16;
  }
}

}  // namespace

cudaError_t launch_route_prepass(const Problem& p, const WsPtrs& ws, const float* tau, uint32_t* mask,
                                 cudaStream_t stream, int* n_launches) {
  const dim3 grid(ceil_div(p.Nk, kProxyCols), ceil_div(p.Nq, kProxyRows), p.BH);
  if (n_launches) *n_launches += 1;
  return launch_after(mask_prepass_kernel, grid, 256, kProxySmem, kProxySmem, 0, stream, ws.qbar, ws.kc, tau, p.forced, mask, p.Nq, p.Nk,
                      p.d, p.scale);
}

}  // namespace sol
