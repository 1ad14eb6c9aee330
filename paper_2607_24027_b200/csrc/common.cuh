// Shared declarations of the Sol-Attn CUDA path: problem description, workspace layout,
// launch prototypes.  Nothing here is used by the CPU oracle.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "sol_attn.h"

namespace sol {

constexpr int kStatusWords = 16;      // int32 words at the start of the workspace
constexpr int kStatusDevice = 0;      // word 0: device status (0 ok, SOL_ERR_DEVICE_TIMEOUT ...)
constexpr int kStatusDetail = 1;      // word 1: where a bounded wait gave up (debug aid)
constexpr int kStatusTileCounter = 2; // word 2: persistent-kernel work counter

__host__ __device__ inline int ceil_div(int a, int b) { return (a + b - 1) / b; }
inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Where element (b, h, n, 0) of q, k, v and out sits (all four share one layout): element strides
// between consecutive tokens, heads and batches.  A token's d channels are always contiguous.
struct Strides {
  long long row, head, batch;
  int H;
  __host__ __device__ size_t base(int bh) const {
    const int b = bh / H;
    return (size_t)b * (size_t)batch + (size_t)(bh - b * H) * (size_t)head;
  }
};

// One attention problem and where its pre-attention results live.
struct Problem {
  int B, H, N, d, block_q, block_k;
  int BH, Nq, Nk;
  int call_heads;    // BH of the whole call, of which this may be a group of heads: what a choice between kernels goes by
  float scale;       // logit scale
  float beta;        // standardized cutoff of Eq. (4)
  int mode;          // SOL_MODE_*
  int estimator;     // SOL_EST_*: how sigma_i is obtained
  const uint8_t* forced;   // device [Nk] or null: key blocks that always go to the exact branch
  Strides st;              // SOL_LAYOUT_*: strides of q, k, v, out
  int routing;             // SOL_ROUTING_*: where the comparison of Eq. (4) is evaluated
};

// Dense mode does not depend on the block size: two query tiles of 128 rows per CTA (fwd_sm100_dense.cu), or the kernel for
// the block size?  All tiles cost the same, so a call is done in rounds of one tile per SM, or of one pair of tiles.
//   128-token blocks (fwd_sm100.cu, one tile): a pair takes as long as 1.97 single tiles at d = 128 and 1.78 at d = 64.
//     d = 128, us with single tiles / pairs: 2 x 4096 tokens (rounds 1 / 1) 39 / 68; 24 x 1024 (2 / 1) 28.3 / 24.6;
//     24 x 2048 (3 / 2) 60 / 73; 24 x 4096 (6 / 3) 227 / 222; 30 x 4096 (7 / 4) 269 / 282; 12 x 11 160 (8 / 4) 773 / 744;
//     24 x 8500 (11 / 6) 869 / 890; 40 x 8192 (18 / 9) 1341 / 1304.
//     d = 64: 12 x 4096 (3 / 2) 101 / 115; 24 x 4096 (6 / 3) 188 / 169; 30 x 4096 (7 / 4) 221 / 221; 40 x 16 000 (34 / 18)
//     3918 / 3695.
//   64-token blocks: up to one block per SM fwd_sm100.cu (2 x 4096 tokens, d = 64 50 / 60, d = 128 56 / 68; 148 blocks, d = 64
//     56 / 69).  Above that always pairs: fwd_sm100_b64.cu, which also takes 256 rows at a time but tiles of 64 keys, has no
//     dense mode, in which it took 1.03 to 1.18 times as long (150 blocks, d = 64 80 / 70 us; 24 x 4096 tokens 192 / 169;
//     40 x 16 000 3965 / 3690; d = 128 12 x 4096 140 / 135).
inline bool dense_in_pairs(int BH, int N, int d, int block_k, int sms) {
  if (block_k == 64) return (long long)BH * ceil_div(N, 64) > sms;
  const long long tiles = (long long)BH * ceil_div(N, 128), pairs = (long long)BH * ceil_div(N, 256);
  const long long rounds = (tiles + sms - 1) / sms, pair_rounds = (pairs + sms - 1) / sms;
  return (d == 128 ? 197 : 178) * pair_rounds <= 100 * rounds;
}

// Byte offsets into the workspace (all multiples of 1024).
struct WsLayout {
  size_t status;  // int32[kStatusWords]
  size_t qbar;    // fp32 [BH][Nq][d]   mean of each query block        (Eq. 3)
  size_t kc;      // fp32 [BH][Nk][d]   mean of each key block          (Eq. 3)
  size_t vc;      // fp32 [BH][Nk][d]   sum of each value block         (before Eq. 9)
  size_t kcb;     // bf16 [BH][Nk][d]   KC rounded, MMA operand of the approximate branch
  size_t vmb;     // bf16 [BH][Nk][d]   VC / n_j rounded, MMA operand of the approximate branch
  size_t mk;      // fp32 [BH][d]       diagonal estimator: first moment of the pooled keys
  size_t vk;      // fp32 [BH][d]       diagonal estimator: channel variances of the pooled keys
  size_t mu, sigma, tau;  // fp32 [BH][Nq] each (Eq. 4)
  size_t total;
};

inline WsLayout make_layout(int BH, int Nq, int Nk, int d) {
  WsLayout w{};
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 1024); return o; };
  w.status = take(sizeof(int32_t) * kStatusWords);
  w.qbar = take(sizeof(float) * (size_t)BH * Nq * d);
  w.kc = take(sizeof(float) * (size_t)BH * Nk * d);
  w.vc = take(sizeof(float) * (size_t)BH * Nk * d);
  w.kcb = take(2 * (size_t)BH * Nk * d);
  w.vmb = take(2 * (size_t)BH * Nk * d);
  w.mk = take(sizeof(float) * (size_t)BH * d);
  w.vk = take(sizeof(float) * (size_t)BH * d);
  w.mu = take(sizeof(float) * (size_t)BH * Nq);
  w.sigma = take(sizeof(float) * (size_t)BH * Nq);
  w.tau = take(sizeof(float) * (size_t)BH * Nq);
  w.total = off;
  return w;
}

// Device pointers handed to the kernels.
struct WsPtrs {
  int32_t* status;
  float *qbar, *kc, *vc;
  __nv_bfloat16 *kcb, *vmb;
  float *mk, *vk, *mu, *sigma, *tau;
};

inline WsPtrs make_ptrs(void* base, const WsLayout& w) {
  char* b = static_cast<char*>(base);
  WsPtrs p;
  p.status = reinterpret_cast<int32_t*>(b + w.status);
  p.qbar = reinterpret_cast<float*>(b + w.qbar);
  p.kc = reinterpret_cast<float*>(b + w.kc);
  p.vc = reinterpret_cast<float*>(b + w.vc);
  p.kcb = reinterpret_cast<__nv_bfloat16*>(b + w.kcb);
  p.vmb = reinterpret_cast<__nv_bfloat16*>(b + w.vmb);
  p.mk = reinterpret_cast<float*>(b + w.mk);
  p.vk = reinterpret_cast<float*>(b + w.vk);
  p.mu = reinterpret_cast<float*>(b + w.mu);
  p.sigma = reinterpret_cast<float*>(b + w.sigma);
  p.tau = reinterpret_cast<float*>(b + w.tau);
  return p;
}

// The kernels of one call follow each other on a stream.  A kernel launched with `launch_after` may start while the
// one before it is still running: its blocks are put in place and set up their barriers and tables, then wait in
// kernel_wait() until the earlier grid has finished and its writes are visible.  Every block calls kernel_wait()
// before it touches global memory, so a kernel that has finished has seen its predecessor finish too.
// kernel_release() lets the next such kernel start before the caller's grid drains; it promises nothing about data.
// Only the small threshold kernel calls it, whose blocks leave room on an SM for the fused kernel's: a release in the
// large pre-attention kernels makes their successors' blocks take up slots their own later blocks need (re-thresholding
// 40 heads of 591 blocks and its bits: 145 us if both kernels release, 92.2 if the threshold kernel does, 91.7 without; 40 heads of
// 256 blocks 56 / 40.5 / 40.4).  A call on 2 heads x 1024 tokens: 22.5 us with plain launches, 18.4 us so.
#ifdef __CUDACC__
__device__ __forceinline__ void kernel_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void kernel_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// `smem`: dynamic shared memory of this launch; `smem_most`: of any launch of the kernel.  The limit is state of the function,
// which other host threads may be launching too, so it never follows a call's own size.
template <class... P, class... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, int threads, size_t smem, size_t smem_most, int cluster,
                         cudaStream_t stream, A... args) {
  cudaError_t e = cudaSuccess;
  // (48 KB is the default limit for static and dynamic shared memory together)
  if (smem_most > 32 * 1024)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_most);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2] = {};
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 0 ? 2 : 1;
  e = cudaLaunchKernelEx(&cfg, kernel, args...);
  return e != cudaSuccess ? e : cudaGetLastError();
}
#endif

// Host-side helpers shared by the files that implement entry points (defined in api.cu).
void count_launches(int n);            // adds to the library's launch counter (sol_attn_launch_count)
sol_status_t check_device_arch();      // SOL_OK on compute capability 10.x, else SOL_ERR_UNSUPPORTED_ARCH

// ---- launchers (each returns the cudaError_t of its launches; all work goes to `stream`) ----

// Pooling pre-pass: Qbar, KC, VC (+ bf16 operand copies).  q may be null.  The status words from `zero_from` on
// are zeroed along the way (kStatusWords: none).
cudaError_t launch_pool(const Problem& p, const __nv_bfloat16* q, const __nv_bfloat16* k,
                        const __nv_bfloat16* v, const WsPtrs& ws, int zero_from, cudaStream_t stream, int* n_launches);

// Pooled-key moments (Eq. 5) and per-query-block mu, sigma, tau (Eq. 4).
cudaError_t launch_thresholds(const Problem& p, const WsPtrs& ws, cudaStream_t stream, int* n_launches);

// Routing pre-pass (SOL_ROUTING_PREPASS): one decision bit per (query block, key block) into `mask`.
cudaError_t launch_route_prepass(const Problem& p, const WsPtrs& ws, const float* tau, uint32_t* mask,
                                 cudaStream_t stream, int* n_launches);

// Fused forward, warp-level mma.sync implementation (all supported shapes).
cudaError_t launch_fwd_mma_sync(const Problem& p, const __nv_bfloat16* q, const __nv_bfloat16* k,
                                const __nv_bfloat16* v, __nv_bfloat16* out, const WsPtrs& ws,
                                const float* tau, int32_t* counts, uint32_t* mask_out,
                                cudaStream_t stream, int* n_launches);

// Fused forward, TMA + tcgen05 + TMEM implementation (d in {64, 128}, block_q = block_k in {64, 128}).
bool fwd_sm100_supports(const Problem& p);
// Test hook: SM clocks after which the kernel's bounded waits give up (<= 0: the default) and the tile
// whose P V completion signal each CTA leaves out (< 0: none); applies to the following launches.
void fwd_sm100_set_wait(long long wait_cycles, int withhold_tile);
cudaError_t launch_fwd_sm100(const Problem& p, const __nv_bfloat16* q, const __nv_bfloat16* k,
                             const __nv_bfloat16* v, __nv_bfloat16* out, const WsPtrs& ws,
                             const float* tau, int32_t* counts, uint32_t* mask_out,
                             cudaStream_t stream, int* n_launches);

}  // namespace sol
