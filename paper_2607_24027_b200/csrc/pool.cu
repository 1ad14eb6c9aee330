// Pre-attention pass of Sol-Attn: block pooling (Eq. 3 and the summed values defined before
// Eq. 9), pooled-key moments (Eq. 5) and per-query-block thresholds (Eq. 4).
//
// The pooling kernel is HBM-bound: it reads q, k and v exactly once with 16-byte loads and
// writes a few MB of pooled vectors.  The moment / threshold kernels touch only pooled data.
#include <cooperative_groups.h>

#include <type_traits>

#include "common.cuh"

namespace sol {
namespace {

constexpr int kPoolThreads = 256;

struct alignas(16) Bf16x8 { __nv_bfloat162 v[4]; };

// One CTA pools one block of one tensor.  A row of d bf16 is covered by d/8 threads with one
// 16-byte load each; the 256 threads form 256/(d/8) row groups that stride over the block's
// rows; partial sums are combined through shared memory.
//   kind 0: q  -> qbar (mean)
//   kind 1: k  -> kc (mean, fp32) and kcb (mean, bf16)
//   kind 2: v  -> vc (sum, fp32)  and vmb (mean, bf16)
template <int D>
__global__ void __launch_bounds__(kPoolThreads)
pool_kernel(const __nv_bfloat16* __restrict__ q, const __nv_bfloat16* __restrict__ k,
            const __nv_bfloat16* __restrict__ v, WsPtrs ws, Strides st, int N, int block_q, int block_k,
            int Nq, int Nk, int first_kind, int zero_from) {
  constexpr int TPR = D / 8;                    // threads per row
  constexpr int RG = kPoolThreads / TPR;        // row groups
  __shared__ float partial[RG][D];

  // the call's status words, which the fused kernel behind this one counts in
  if (blockIdx.x == 0 && threadIdx.x >= zero_from && threadIdx.x < kStatusWords) ws.status[threadIdx.x] = 0;

  // blockIdx.x enumerates, per (batch, head): Nq query blocks (if q is pooled), Nk key blocks,
  // Nk value blocks.
  const int per_bh = (first_kind == 0 ? Nq : 0) + 2 * Nk;
  const int bh = blockIdx.x / per_bh;
  int r = blockIdx.x - bh * per_bh;
  int kind, blk;
  if (first_kind == 0 && r < Nq) { kind = 0; blk = r; }
  else {
    if (first_kind == 0) r -= Nq;
    if (r < Nk) { kind = 1; blk = r; } else { kind = 2; blk = r - Nk; }
  }
  const int bs = (kind == 0) ? block_q : block_k;
  const __nv_bfloat16* src = (kind == 0) ? q : (kind == 1 ? k : v);
  const int row0 = blk * bs;
  const int nvalid = min(bs, N - row0);
  const __nv_bfloat16* base = src + st.base(bh) + (size_t)row0 * st.row;

  const int tc = threadIdx.x % TPR;             // which 8-channel group of the row
  const int g = threadIdx.x / TPR;              // row group
  float acc[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c] = 0.f;

  int row = g;
  // four independent 16-byte loads in flight per thread
  for (; row + 3 * RG < nvalid; row += 4 * RG) {
    Bf16x8 x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      x[u] = *reinterpret_cast<const Bf16x8*>(base + (size_t)(row + u * RG) * st.row + tc * 8);
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float2 f = __bfloat1622float2(x[u].v[c]);
        acc[2 * c] += f.x;
        acc[2 * c + 1] += f.y;
      }
  }
  for (; row < nvalid; row += RG) {
    Bf16x8 x = *reinterpret_cast<const Bf16x8*>(base + (size_t)row * st.row + tc * 8);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float2 f = __bfloat1622float2(x.v[c]);
      acc[2 * c] += f.x;
      acc[2 * c + 1] += f.y;
    }
  }
#pragma unroll
  for (int c = 0; c < 8; ++c) partial[g][tc * 8 + c] = acc[c];
  __syncthreads();

  if (threadIdx.x < D) {
    const int c = threadIdx.x;
    float s = 0.f;
#pragma unroll 8
    for (int gg = 0; gg < RG; ++gg) s += partial[gg][c];
    const float mean = s / (float)nvalid;
    if (kind == 0) {
      ws.qbar[((size_t)bh * Nq + blk) * D + c] = mean;
    } else if (kind == 1) {
      const size_t o = ((size_t)bh * Nk + blk) * D + c;
      ws.kc[o] = mean;
      ws.kcb[o] = __float2bfloat16_rn(mean);
    } else {
      const size_t o = ((size_t)bh * Nk + blk) * D + c;
      ws.vc[o] = s;
      ws.vmb[o] = __float2bfloat16_rn(mean);
    }
  }
}

__device__ __forceinline__ float4 add4(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 sub4(float4 a, float4 b) { return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }

// mu, sigma and tau of one query block, from its raw products.
__device__ __forceinline__ void store_threshold(const WsPtrs& ws, size_t o, float mu, float sigma, float beta) {
  ws.mu[o] = mu;
  ws.sigma[o] = sigma;
  ws.tau[o] = isinf(beta) ? beta : fmaf(beta, sigma, mu);   // +inf: route nothing, -inf: route everything
}

// Thresholds of a head with few pooled keys (Nk <= kSmallKeys), in one launch.  A CTA takes 16 query blocks
// of one head, with all pooled keys of the head in shared memory: mean, then centred keys x_j = KC_j - m_K,
// then the row statistics straight from the centred scores,
//   mu_i = s Qbar_i . m_K,   sigma_i^2 = s^2 (1/Nk) sum_j (Qbar_i . x_j)^2,
// which is Eq. (4)'s own definition (and Eq. 5's quadratic form with the sums exchanged).  With kDiag the
// diagonal estimator: sigma_i^2 = s^2 (Qbar_i o Qbar_i) . v_K, v_K = (1/Nk) sum_j x_j o x_j.
//
// These sizes are bound by latency: a launch and a few dependent passes over a few KB.  24 heads of 32 key and
// 32 query blocks, d = 128: 6.4 us, where the three kernels of the moments (mean, second moment, quadratic
// form) took 42 us and two more launches.  Its work grows with Nq Nk, that of the second moment with
// (Nq + Nk) d, so the line lies at Nk = d.
constexpr int kSmallKeys = 128, kSmallRows = 16;

template <int D, bool kDiag>
__global__ void __launch_bounds__(256) thresholds_small_kernel(WsPtrs ws, int Nq, int Nk, float scale, float beta) {
  constexpr int LD = D + 4;                      // rows 4 banks apart: 16-byte reads of eight rows do not collide
  constexpr int G = 256 / D;                     // threads per channel
  extern __shared__ __align__(16) float smem_f[];
  float* ks = smem_f;                            // [Nk][LD]
  __shared__ __align__(16) float qs[kSmallRows][LD];
  __shared__ float part[G][D], mean_s[D], var_s[kDiag ? D : 1];
  const int bh = blockIdx.y, i0 = blockIdx.x * kSmallRows, tid = threadIdx.x;
  const float* kc = ws.kc + (size_t)bh * Nk * D;
  const float* qb = ws.qbar + ((size_t)bh * Nq + i0) * D;
  const int nq = min(kSmallRows, Nq - i0);
  kernel_wait();
  kernel_release();
#pragma unroll 4
  for (int e = tid; e < Nk * (D / 4); e += 256)
    *reinterpret_cast<float4*>(ks + (e / (D / 4)) * LD + (e % (D / 4)) * 4) = reinterpret_cast<const float4*>(kc)[e];
  for (int e = tid; e < kSmallRows * (D / 4); e += 256)
    *reinterpret_cast<float4*>(&qs[e / (D / 4)][(e % (D / 4)) * 4]) =
        e / (D / 4) < nq ? reinterpret_cast<const float4*>(qb)[e] : make_float4(0.f, 0.f, 0.f, 0.f);
  __syncthreads();
  const int c = tid % D, g = tid / D;
  auto total = [&](float s) {                    // sum over the G threads of a channel, in a fixed order
    part[g][c] = s;
    __syncthreads();
    float r = 0.f;
#pragma unroll
    for (int x = 0; x < G; ++x) r += part[x][c];
    __syncthreads();
    return r;
  };
  float s = 0.f;
#pragma unroll 8
  for (int j = g; j < Nk; j += G) s += ks[j * LD + c];
  const float m = total(s) / (float)Nk;
  float sq = 0.f;
#pragma unroll 8
  for (int j = g; j < Nk; j += G) {
    const float x = ks[j * LD + c] - m;
    if constexpr (kDiag) sq = fmaf(x, x, sq);
    else ks[j * LD + c] = x;
  }
  if constexpr (kDiag) {
    const float v = total(sq) / (float)Nk;
    if (g == 0) var_s[c] = v;
  }
  if (g == 0) mean_s[c] = m;
  __syncthreads();
  const int row = tid / 16, tx = tid % 16;
  float quad = 0.f, dotm = 0.f;
  if constexpr (!kDiag) {
    const float4* q4 = reinterpret_cast<const float4*>(qs[row]);
    for (int j = tx; j < Nk; j += 32) {          // two keys at a time
      const bool two = j + 16 < Nk;
      const float4* ka = reinterpret_cast<const float4*>(ks + j * LD);
      const float4* kb = two ? ka + 16 * (LD / 4) : ka;
      float2 a0 = make_float2(0.f, 0.f), a1 = a0, b0 = a0, b1 = a0;
#pragma unroll 8
      for (int p = 0; p < D / 4; ++p) {
        const float4 q = q4[p], x = ka[p], y = kb[p];
        a0 = __ffma2_rn(make_float2(q.x, q.y), make_float2(x.x, x.y), a0);
        a1 = __ffma2_rn(make_float2(q.z, q.w), make_float2(x.z, x.w), a1);
        b0 = __ffma2_rn(make_float2(q.x, q.y), make_float2(y.x, y.y), b0);
        b1 = __ffma2_rn(make_float2(q.z, q.w), make_float2(y.z, y.w), b1);
      }
      const float sa = (a0.x + a0.y) + (a1.x + a1.y), sb = (b0.x + b0.y) + (b1.x + b1.y);
      quad = fmaf(sa, sa, quad);
      if (two) quad = fmaf(sb, sb, quad);
    }
    quad /= (float)Nk;
  }
#pragma unroll
  for (int p = 0; p < D / 16; ++p) {
    const float q = qs[row][tx + 16 * p];
    dotm = fmaf(q, mean_s[tx + 16 * p], dotm);
    if constexpr (kDiag) quad = fmaf(q * q, var_s[tx + 16 * p], quad);
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) {
    quad += __shfl_xor_sync(0xffffffffu, quad, o);
    dotm += __shfl_xor_sync(0xffffffffu, dotm, o);
  }
  if (tx == 0 && row < nq)
    store_threshold(ws, (size_t)bh * Nq + i0 + row, scale * dotm, scale * sqrtf(fmaxf(quad, 0.f)), beta);
}

// Thresholds of a head with many pooled keys, in one launch: the moments m_K and
//   C_K = (1/Nk) sum_j (KC_j - m_K)^T (KC_j - m_K)
// (the bracket of Eq. 5 with the mu_i^2 term already folded in, which avoids the cancellation of the
// uncentred form in fp32), then per query block mu_i = s Qbar_i . m_K, sigma_i^2 = s^2 Qbar_i C_K Qbar_i^T.
//
// A thread-block cluster takes one head.  How many CTAs it has depends on how many heads the call has, but nothing
// that is summed does, so that a head's thresholds are the same in every call it is part of:
//   m_K   eight slices of the keys, summed in order whichever CTA summed which;
//   C_K   is cut by its entries, not by the keys: it is symmetric, and of its 4 x 4 blocks the ten on and above the
//         diagonal are dealt out to the CTAs.  Every entry is the sum of four chains of FMAs, one over every fourth key
//         (one chain over all keys, as a single CTA per head has it when the keys are dealt out, has a quarter more error).
// Then every CTA gathers the whole C_K and forms Y = Qbar C_K for its share of the query blocks, up to 88 in one step (with
// two CTAs per SM that is the largest `work` area there is room for).
constexpr int kMomentRows = 88, kMeanSlices = 8;

template <int D>
constexpr int kMomentChunk = D == 128 ? 32 : 64; // keys in shared memory, twice
template <int D>
constexpr int kKeyLd = D + 16;                   // floats from one to the next: neighbours half a bank cycle apart, see below

template <int D>
constexpr size_t moments_smem() {                // C_K, then (in turn) partial sums / two chunks of keys / pooled queries
  constexpr size_t rows = sizeof(float) * kMomentRows * D, chunks = sizeof(float) * 2 * kMomentChunk<D> * kKeyLd<D>;
  constexpr size_t sums = sizeof(float) * kMeanSlices * 256 * 4;
  return sizeof(float) * D * D + (rows > chunks ? (rows > sums ? rows : sums) : (chunks > sums ? chunks : sums));
}

template <int D>
__global__ void __launch_bounds__(256, 2) thresholds_moments_kernel(WsPtrs ws, int Nq, int Nk, float scale, float beta) {
  constexpr int T = D / 16;                      // columns of Y per thread (8 or 4)
  constexpr int P4 = D / 4;                      // 16-byte pieces of a row
  constexpr int E = D / 4, kBlocks = 10;         // edge of a block of C_K, blocks on and above the diagonal
  constexpr int M = E / 4;                       // rows and columns of a block per thread (8 or 4)
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int n_cta = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  extern __shared__ __align__(16) float smem_f[];
  float* cov = smem_f;                           // [D][D]
  float* work = smem_f + D * D;
  __shared__ __align__(16) float sum_s[kMeanSlices][D], mean_s[D];
  const int bh = blockIdx.y, tid = threadIdx.x;
  const int ty = tid / 16, tx = tid % 16;
  const int piece = tid % P4;                    // (256 is a multiple of P4: the same piece of every row it touches)
  const float4* kc4 = reinterpret_cast<const float4*>(ws.kc + (size_t)bh * Nk * D);
  float4* work4 = reinterpret_cast<float4*>(work);
  auto sync = [&] {
    if (n_cta > 1) cluster.sync();
    else __syncthreads();
  };
  kernel_wait();

  // ---- m_K
  {
    const int per = ceil_div(Nk, kMeanSlices);
    for (int y = rank; y < kMeanSlices; y += n_cta) {
      const int end = min(Nk, (y + 1) * per);
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
      for (int j = y * per + tid / P4; j < end; j += 256 / P4) x = add4(x, kc4[(size_t)j * P4 + piece]);
      work4[y * 256 + tid] = x;
    }
    __syncthreads();
    for (int y = rank; y < kMeanSlices; y += n_cta)
      if (tid < D) {
        float r = 0.f;
#pragma unroll
        for (int g = 0; g < 256 / P4; ++g) r += work[(y * 256 + g * P4) * 4 + tid];
        sum_s[y][tid] = r;
      }
    sync();
    if (tid < D) {
      float x[kMeanSlices], r = 0.f;
#pragma unroll
      for (int y = 0; y < kMeanSlices; ++y) x[y] = cluster.map_shared_rank(&sum_s[y][0], y % n_cta)[tid];
#pragma unroll
      for (int y = 0; y < kMeanSlices; ++y) r += x[y];
      mean_s[tid] = r / (float)Nk;
    }
    __syncthreads();
  }

  // ---- this CTA's blocks of C_K, in passes over the keys of up to four blocks.  A block belongs to 64 threads, or to 128
  //      or all 256 where a pass has fewer: 16 threads share it in patches of M x M entries, rows r0 + x (+ 16) and columns
  //      c0 + y (+ 16), each for every fourth key, and the patches are cut into `parts` of R rows.  The two quarters of the
  //      keys that a warp works on lie in neighbouring rows, 16 floats off in the banks: no conflicts.
  const float4 m4 = *reinterpret_cast<const float4*>(mean_s + 4 * piece);
  const int quarter = tid % 64 / 16, r0 = tid % 16 / 4 * 4, c0 = tid % 4 * 4;
  constexpr int LD = kKeyLd<D>, kChunk = kMomentChunk<D>;
  const int n_chunks = ceil_div(Nk, kChunk);
  constexpr int kPre = kChunk * P4 / 256;        // pieces of a chunk per thread
  float4 pre[kPre];
  auto fetch = [&](int chunk) {
#pragma unroll
    for (int i = 0; i < kPre; ++i) {
      const int j = chunk * kChunk + (tid + 256 * i) / P4;
      pre[i] = j < Nk ? kc4[(size_t)j * P4 + piece] : m4;
    }
  };
  auto put = [&](int chunk) {                    // centred; keys past the last one are zero
    float* to = work + (chunk & 1) * kChunk * LD + 4 * piece;
#pragma unroll
    for (int i = 0; i < kPre; ++i) *reinterpret_cast<float4*>(to + (tid + 256 * i) / P4 * LD) = sub4(pre[i], m4);
  };
  auto block_row = [](int b) { return (b >= 4) + (b >= 7) + (b >= 9); };
  auto block_col = [](int b, int bi) { return b - (4 * bi - bi * (bi - 1) / 2) + bi; };
  auto pass = [&](auto r_c, int first) {         // blocks first + slot n_cta + rank
    constexpr int R = decltype(r_c)::value, kParts = M / R, kSlots = 4 / kParts;
    const int group = tid / 64, part = group % kParts, b = first + group / kParts * n_cta + rank;
    const int bi = block_row(b), bj = block_col(b, bi);
    const int rp = r0 + part * R / 4 * 16 + part * R % 4;    // first row of the part
    float2 acc[R][M / 2];
#pragma unroll
    for (int x = 0; x < R; ++x)
#pragma unroll
      for (int y = 0; y < M / 2; ++y) acc[x][y] = make_float2(0.f, 0.f);
    fetch(0);
    put(0);
    __syncthreads();
    for (int t = 0; t < n_chunks; ++t) {
      if (t + 1 < n_chunks) fetch(t + 1);
      if (b < kBlocks) {
        const float* row = work + ((t & 1) * kChunk + quarter) * LD + bi * E + rp;
        const float* col = work + ((t & 1) * kChunk + quarter) * LD + bj * E + c0;
#pragma unroll 2
        for (int j = 0; j < kChunk; j += 4) {
          float u[R], v[M];
          if constexpr (R >= 4) {
#pragma unroll
            for (int h = 0; h < R / 4; ++h)
              *reinterpret_cast<float4*>(u + 4 * h) = *reinterpret_cast<const float4*>(row + j * LD + 16 * h);
          } else if constexpr (R == 2) {
            *reinterpret_cast<float2*>(u) = *reinterpret_cast<const float2*>(row + j * LD);
          } else {
            u[0] = row[j * LD];
          }
#pragma unroll
          for (int h = 0; h < M / 4; ++h)
            *reinterpret_cast<float4*>(v + 4 * h) = *reinterpret_cast<const float4*>(col + j * LD + 16 * h);
#pragma unroll
          for (int x = 0; x < R; ++x)
#pragma unroll
            for (int y = 0; y < M / 2; ++y)
              acc[x][y] = __ffma2_rn(make_float2(u[x], u[x]), make_float2(v[2 * y], v[2 * y + 1]), acc[x][y]);
        }
      }
      if (t + 1 < n_chunks) put(t + 1);
      __syncthreads();
    }
    // the quarters: 0 + 1 and 2 + 3 within a warp, the two sums through shared memory ([2][slot][E][E])
#pragma unroll
    for (int x = 0; x < R; ++x)
#pragma unroll
      for (int y = 0; y < M / 2; ++y) {
        acc[x][y].x += __shfl_xor_sync(0xffffffffu, acc[x][y].x, 16);
        acc[x][y].y += __shfl_xor_sync(0xffffffffu, acc[x][y].y, 16);
      }
    if (quarter % 2 == 0) {
      float* to = work + ((quarter / 2 * kSlots + group / kParts) * E + rp) * E + c0;
#pragma unroll
      for (int x = 0; x < R; ++x)
#pragma unroll
        for (int h = 0; h < M / 4; ++h)
          *reinterpret_cast<float4*>(to + (x / 4 * 16 + x % 4) * E + 16 * h) =
              make_float4(acc[x][2 * h].x, acc[x][2 * h].y, acc[x][2 * h + 1].x, acc[x][2 * h + 1].y);
    }
    __syncthreads();
    constexpr int kPieces = E * E / 4;
    for (int e = tid; e < kSlots * kPieces; e += 256) {
      const int bb = first + e / kPieces * n_cta + rank, at = e % kPieces;
      if (bb >= kBlocks) break;                  // (and so are the slots behind it)
      float4 x = add4(work4[e], work4[kSlots * kPieces + e]);
      const float n = (float)Nk;
      x.x /= n; x.y /= n; x.z /= n; x.w /= n;
      const int xi = block_row(bb), xj = block_col(bb, xi), i = xi * E + at / (E / 4), j = xj * E + at % (E / 4) * 4;
      *reinterpret_cast<float4*>(cov + i * D + j) = x;
      if (xi != xj) {                            // the mirror image below the diagonal
        cov[j * D + i] = x.x;
        cov[(j + 1) * D + i] = x.y;
        cov[(j + 2) * D + i] = x.z;
        cov[(j + 3) * D + i] = x.w;
      }
    }
    __syncthreads();
    return first + kSlots * n_cta;
  };
  for (int first = 0; first < kBlocks;) {
    const int per = ceil_div(kBlocks - first, n_cta);          // blocks that this CTA may still have
    if (per > 2) first = pass(std::integral_constant<int, M>{}, first);
    else if (per == 2) first = pass(std::integral_constant<int, M / 2>{}, first);
    else first = pass(std::integral_constant<int, M / 4>{}, first);
  }
  sync();
  if (n_cta > 1) {
    // gather the other CTAs' blocks
#pragma unroll 8
    for (int e = tid; e < D * P4; e += 256) {
      const int x = e / P4 / E, y = piece * 4 / E, bi = min(x, y), bj = max(x, y);
      const int owner = (4 * bi - bi * (bi - 1) / 2 + bj - bi) % n_cta;
      if (owner != rank)
        reinterpret_cast<float4*>(cov)[e] = reinterpret_cast<const float4*>(cluster.map_shared_rank(cov, owner))[e];
    }
    cluster.sync();                              // a CTA may leave once its blocks are read
  }

  // ---- Y = Qbar C_K and the row sums of Y o Qbar; thread (ty, tx) owns query blocks ty + 16 a and columns
  //      4 tx + c (+ 64)
  const int per_q = ceil_div(Nq, n_cta);
  const int i_begin = min(Nq, rank * per_q), i_end = min(Nq, i_begin + per_q);
  auto rows = [&](auto a_c, int i0) {
    constexpr int A = decltype(a_c)::value;
    const int nq = min(min(16 * A, kMomentRows), i_end - i0);
#pragma unroll 4
    for (int e = tid; e < nq * P4; e += 256) work4[e] = reinterpret_cast<const float4*>(ws.qbar + ((size_t)bh * Nq + i0) * D)[e];
    __syncthreads();
    const float* q_row[A];                       // (rows past the last repeat it and are not stored)
#pragma unroll
    for (int a = 0; a < A; ++a) q_row[a] = work + min(ty + 16 * a, nq - 1) * D;
    float2 y[A][T / 2];
#pragma unroll
    for (int a = 0; a < A; ++a)
#pragma unroll
      for (int c = 0; c < T / 2; ++c) y[a][c] = make_float2(0.f, 0.f);
    // (unrolled by two, so that one step's reads go beside the other's FMAs: 40 x 591 x 591 blocks 57.7 -> 55.7 us, 80 x 300 59.3 ->
    //  58.0; by four, or with one CTA per SM and its registers, 54 / 72)
#pragma unroll 2
    for (int k = 0; k < D; k += 4) {
      float q[A][4];
#pragma unroll
      for (int a = 0; a < A; ++a)
        *reinterpret_cast<float4*>(q[a]) = *reinterpret_cast<const float4*>(q_row[a] + k);
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        float b[T];
#pragma unroll
        for (int h = 0; h < T / 4; ++h)
          *reinterpret_cast<float4*>(b + 4 * h) = *reinterpret_cast<const float4*>(cov + (k + kk) * D + 64 * h + 4 * tx);
#pragma unroll
        for (int a = 0; a < A; ++a)
#pragma unroll
          for (int c = 0; c < T / 2; ++c)
            y[a][c] = __ffma2_rn(make_float2(q[a][kk], q[a][kk]), make_float2(b[2 * c], b[2 * c + 1]), y[a][c]);
      }
    }
#pragma unroll
    for (int a = 0; a < A; ++a) {
      float quad = 0.f, dotm = 0.f;
#pragma unroll
      for (int c = 0; c < T; ++c) {
        const int at = (c / 4) * 64 + 4 * tx + c % 4;
        const float qv = q_row[a][at];
        quad = fmaf((c & 1) ? y[a][c / 2].y : y[a][c / 2].x, qv, quad);
        dotm = fmaf(qv, mean_s[at], dotm);
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
        quad += __shfl_xor_sync(0xffffffffu, quad, o);
        dotm += __shfl_xor_sync(0xffffffffu, dotm, o);
      }
      if (tx == 0 && ty + 16 * a < nq)
        store_threshold(ws, (size_t)bh * Nq + i0 + ty + 16 * a, scale * dotm, scale * sqrtf(fmaxf(quad, 0.f)), beta);
    }
    __syncthreads();
  };
  for (int i0 = i_begin; i0 < i_end;) {          // a step is as short as what is left
    const int left = i_end - i0;
    if (left > 64) {
      rows(std::integral_constant<int, 6>{}, i0);
      i0 += kMomentRows;
    } else if (left > 32) {
      rows(std::integral_constant<int, 4>{}, i0);
      i0 += 64;
    } else {
      rows(std::integral_constant<int, 2>{}, i0);
      i0 += 32;
    }
  }
}

}  // namespace

cudaError_t launch_pool(const Problem& p, const __nv_bfloat16* q, const __nv_bfloat16* k,
                        const __nv_bfloat16* v, const WsPtrs& ws, int zero_from, cudaStream_t stream, int* n_launches) {
  const int first_kind = q ? 0 : 1;
  const long long blocks = (long long)p.BH * ((q ? p.Nq : 0) + 2LL * p.Nk);
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  if (p.d == 128)
    pool_kernel<128><<<(unsigned)blocks, kPoolThreads, 0, stream>>>(q, k, v, ws, p.st, p.N, p.block_q, p.block_k,
                                                                      p.Nq, p.Nk, first_kind, zero_from);
  else
    pool_kernel<64><<<(unsigned)blocks, kPoolThreads, 0, stream>>>(q, k, v, ws, p.st, p.N, p.block_q, p.block_k,
                                                                     p.Nq, p.Nk, first_kind, zero_from);
  if (n_launches) *n_launches += 1;
  return cudaGetLastError();
}

// Diagonal estimator (appendix, Eq. appendix_diagonal_threshold): only the per-channel variance of
// the pooled keys is kept, v_K = mean_j KC_j o KC_j - m_K o m_K (computed in centred form), and
// sigma_i^2 = s^2 (Qbar_i o Qbar_i) . v_K.  One CTA per (batch, head) writes m_K and v_K.
template <int D>
__global__ void __launch_bounds__(4 * D) key_diag_kernel(WsPtrs ws, int Nk) {
  __shared__ float part[4][D];
  __shared__ float mean_s[D];
  const int bh = blockIdx.x, c = threadIdx.x % D, grp = threadIdx.x / D;
  const float* kc = ws.kc + (size_t)bh * Nk * D;
  float s = 0.f;
  for (int j = grp; j < Nk; j += 4) s += kc[(size_t)j * D + c];
  part[grp][c] = s;
  __syncthreads();
  if (grp == 0) mean_s[c] = ((part[0][c] + part[1][c]) + (part[2][c] + part[3][c])) / (float)Nk;
  __syncthreads();
  const float m = mean_s[c];
  float v = 0.f;
  for (int j = grp; j < Nk; j += 4) {
    const float x = kc[(size_t)j * D + c] - m;
    v = fmaf(x, x, v);
  }
  __syncthreads();
  part[grp][c] = v;
  __syncthreads();
  if (grp == 0) {
    ws.mk[(size_t)bh * D + c] = m;
    ws.vk[(size_t)bh * D + c] = ((part[0][c] + part[1][c]) + (part[2][c] + part[3][c])) / (float)Nk;
  }
}

// One warp per query block: mu_i, sigma_i (diagonal form), tau_i.
template <int D>
__global__ void __launch_bounds__(256) tau_diag_kernel(WsPtrs ws, int Nq, float scale, float beta) {
  const int bh = blockIdx.y;
  const int i = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
  if (i >= Nq) return;
  const float* qb = ws.qbar + ((size_t)bh * Nq + i) * D;
  const float* mk = ws.mk + (size_t)bh * D;
  const float* vk = ws.vk + (size_t)bh * D;
  float quad = 0.f, dotm = 0.f;
#pragma unroll
  for (int c = lane; c < D; c += 32) {
    const float qv = qb[c];
    quad = fmaf(qv * qv, vk[c], quad);
    dotm = fmaf(qv, mk[c], dotm);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    quad += __shfl_xor_sync(0xffffffffu, quad, o);
    dotm += __shfl_xor_sync(0xffffffffu, dotm, o);
  }
  if (lane == 0) {
    store_threshold(ws, (size_t)bh * Nq + i, scale * dotm, scale * sqrtf(fmaxf(quad, 0.f)), beta);
  }
}

// CTAs per head of thresholds_moments_kernel: the size with the least time.  `cycles` is a CTA's time in thousands (591 x 591
// blocks, d = 128; other sizes are in much the same proportions).  As many CTAs as find an SM of their own run at that pace:
// clusters of 1 and 2 fill the GPU, clusters of 3 to 6 about 17/20 of it, and of clusters of 8 no more than 14 are placed at
// once.  Two CTAs on an SM share its FMA pipes and take 1.8 times as long.  The table was taken before the quadratic form's loop was
// unrolled, which made the larger clusters more alike (a CTA's time, us of a call: 8 31.6, 6 and 5 38, 4 45, 3 55, 2 78, 1 132); the
// sizes taken are still the best of all at each of these: us with the size taken / others, d = 128: 40 heads x 591 blocks
// (3) 55.7 / 5: 61, 6: 69, 4: 76, 2: 79; 16 x 591 (6) 38.8 / 4: 45, 8: 50; 28 x 591 (4) 45.6 / 8: 51, 3: 56; 48 x 300 (5) 36 / 2: 47;
// 80 x 300 (3) 58 / 5: 60, 2: 74; 100 x 160 (2) 45.3 / 1: 47; d = 64: 40 x 591 (3) 25.9 / 5: 27.5; 24 x 591 (5) 19.9 / 4: 21.
static int cluster_size(int heads, int sms) {
  struct { int n, cycles; } const sizes[] = {{8, 46}, {6, 53}, {5, 58}, {4, 82}, {3, 95}, {2, 141}, {1, 268}};
  int best = 1;
  long long least = -1;
  for (const auto& s : sizes) {
    const long long ctas = (long long)heads * s.n;
    const long long fit = s.n == 8 ? 8 * (14 * sms / 148) : (s.n > 2 ? sms * 17 / 20 : sms);
    if (s.n > 1 && ctas > 2 * fit) continue;     // (would wait for its turn)
    const long long time = ctas <= fit ? 10LL * s.cycles : 18LL * s.cycles;
    if (least < 0 || time < least) { least = time; best = s.n; }
  }
  return best;
}

template <int D>
static cudaError_t thresholds_impl(const Problem& p, const WsPtrs& ws, cudaStream_t stream, int* n_launches) {
  const bool diag = p.estimator == SOL_EST_DIAGONAL;
  if (p.Nk <= kSmallKeys) {
    if (n_launches) *n_launches += 1;
    return launch_after(diag ? thresholds_small_kernel<D, true> : thresholds_small_kernel<D, false>,
                        dim3(ceil_div(p.Nq, kSmallRows), p.BH), 256, sizeof(float) * p.Nk * (D + 4),
                        sizeof(float) * kSmallKeys * (D + 4), 0, stream, ws, p.Nq, p.Nk, p.scale, p.beta);
  }
  if (diag) {
    key_diag_kernel<D><<<p.BH, 4 * D, 0, stream>>>(ws, p.Nk);
    tau_diag_kernel<D><<<dim3(ceil_div(p.Nq, 8), p.BH), 256, 0, stream>>>(ws, p.Nq, p.scale, p.beta);
    if (n_launches) *n_launches += 2;
    return cudaGetLastError();
  }
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int n_cta = cluster_size(p.BH, sms);
  if (n_launches) *n_launches += 1;
  return launch_after(thresholds_moments_kernel<D>, dim3(n_cta, p.BH), 256, moments_smem<D>(), moments_smem<D>(), n_cta, stream, ws, p.Nq, p.Nk,
                      p.scale, p.beta);
}

cudaError_t launch_thresholds(const Problem& p, const WsPtrs& ws, cudaStream_t stream, int* n_launches) {
  return p.d == 128 ? thresholds_impl<128>(p, ws, stream, n_launches)
                    : thresholds_impl<64>(p, ws, stream, n_launches);
}

}  // namespace sol
