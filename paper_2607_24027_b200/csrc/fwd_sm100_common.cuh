// What the tcgen05 forward kernels (fwd_sm100.cu: 128-token blocks, fwd_sm100_b64.cu: 64-token blocks,
// fwd_sm100_dense.cu: dense mode) have in common: launch parameters, the failure flag and a few TMEM / descriptor helpers.
#pragma once

#include "common.cuh"
#include "ptx_sm100.cuh"
#include "tmap.cuh"

namespace sol {
namespace fwd {

using namespace ptx;

constexpr int kRowsQ = 128;                      // rows of the query tile fed to the tensor core
constexpr int kThreads = 384;
constexpr int kWarpRouter = 8, kWarpProducer = 9;
constexpr int kTmemCols = 512;
constexpr float kRescaleThreshold = 8.0f;        // log2 units

struct Params {
  const float* qbar;            // [BH][Nq][d]
  const float* kc;              // [BH][Nk][d]
  const float* tau;             // [BH][Nq]
  __nv_bfloat16* out;
  int32_t* counts;
  uint32_t* mask_out;
  int32_t* status;              // workspace status words
  int N, Nq, Nk, total_work, mode;
  float scale;
  const uint8_t* forced;        // [Nk] or null: key blocks always routed to the exact branch
  Strides st;                   // layout of q, k, v, out
  int rows_inner;               // coordinate order of the q/k/v tensor maps: (c, row, h, b) or (c, h, row, b)
  long long wait_limit;         // SM clocks after which a bounded wait gives up
  int withhold_tile;            // test hook: >= 0: the completion signal of this tile's value GEMM is left out
  int out_aligned32;            // every output row piece starts on a 32-byte boundary (32-byte stores are legal)
  int per_item, items_per_head; // 64-token blocks: query blocks per work item
};

// Test hook (sol_attn_debug_set_wait): the wait limit and the withheld tile of the following launches (fwd_sm100.cu).
extern long long g_wait_limit;
extern int g_withhold_tile;

struct Maps {                   // q, k, v in the caller's layout; KC and mean-V, dense [B][H][Nk][d]
  CUtensorMap q, k, v, kc, vm;
};

template <class S>
__device__ __forceinline__ void flag_abort(S& sm, const Params& p, int where) {
  sm.abort_flag = 1;
  atomicExch(p.status + kStatusDevice, (int)SOL_ERR_DEVICE_TIMEOUT);
  atomicCAS(p.status + kStatusDetail, 0, where);     // keep the first place that gave up
}

// Shared-memory descriptors: the upper word is constant (stride 1024 B between 8-row groups,
// descriptor version, 128-byte swizzle); the lower word is (address >> 4) | (leading offset >> 4) << 16.
__device__ __forceinline__ uint64_t desc_from_lo(uint32_t lo) {
  constexpr uint32_t hi = (1024u >> 4) | (1u << 14) | (2u << 29);
  return ((uint64_t)hi << 32) | lo;
}

template <int N>
__device__ __forceinline__ void tmem_ld_cols(uint32_t taddr, uint32_t* r) {   // N columns, N a multiple of 32
#pragma unroll
  for (int c = 0; c < N; c += 32) tmem_ld_32x32b_x32(taddr + c, *reinterpret_cast<uint32_t(*)[32]>(r + c));
}

// Tensor maps and launch parameters of one problem, K and V tiles of kv_rows keys (everything but the work split and the test hook's state).
inline bool prepare(const Problem& p, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                    __nv_bfloat16* out, const WsPtrs& ws, const float* tau, int32_t* counts, uint32_t* mask_out,
                    int kv_rows, Maps* m, Params* prm) {
  bool rows_inner = true, pooled_inner = true;
  auto user_map = [&](CUtensorMap* t, const void* base, int box_rows) {
    return make_tmap_bf16_4d(t, base, p.B, p.H, p.N, p.d, box_rows, p.st.row, p.st.head, p.st.batch, &rows_inner);
  };
  auto pooled_map = [&](CUtensorMap* t, const void* base) {      // dense [B][H][Nk][d]
    return make_tmap_bf16_4d(t, base, p.B, p.H, p.Nk, p.d, p.block_k, p.d, (long long)p.Nk * p.d,
                             (long long)p.H * p.Nk * p.d, &pooled_inner);
  };
  if (!user_map(&m->q, q, kRowsQ) || !user_map(&m->k, k, kv_rows) || !user_map(&m->v, v, kv_rows) ||
      !pooled_map(&m->kc, ws.kcb) || !pooled_map(&m->vm, ws.vmb) || !pooled_inner)
    return false;
  *prm = Params{};
  prm->qbar = ws.qbar; prm->kc = ws.kc; prm->tau = tau; prm->out = out; prm->counts = counts; prm->mask_out = mask_out;
  prm->status = ws.status; prm->N = p.N; prm->Nq = p.Nq; prm->Nk = p.Nk;
  prm->mode = p.mode; prm->scale = p.scale; prm->forced = p.forced;
  prm->st = p.st; prm->rows_inner = rows_inner ? 1 : 0;
  prm->out_aligned32 = (reinterpret_cast<uintptr_t>(out) % 32 == 0 && (p.st.row * 2) % 32 == 0 &&
                        (p.st.head * 2) % 32 == 0 && (p.st.batch * 2) % 32 == 0) ? 1 : 0;
  return true;
}

inline cudaError_t sm_count(int* sms) {
  int dev = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  return e != cudaSuccess ? e : cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
}

// The 64-token-block kernel's launcher (fwd_sm100_b64.cu); `wait_limit` and `withhold_tile` as in Params.
cudaError_t launch_b64(const Problem& p, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                       __nv_bfloat16* out, const WsPtrs& ws, const float* tau, int32_t* counts, uint32_t* mask_out,
                       long long wait_limit, int withhold_tile, cudaStream_t stream, int* n_launches);

// The dense kernel's launcher (fwd_sm100_dense.cu).
cudaError_t launch_dense(const Problem& p, const __nv_bfloat16* q, const __nv_bfloat16* k, const __nv_bfloat16* v,
                         __nv_bfloat16* out, const WsPtrs& ws, int32_t* counts, uint32_t* mask_out, int sms,
                         long long wait_limit, int withhold_tile, cudaStream_t stream, int* n_launches);

}  // namespace fwd
}  // namespace sol
