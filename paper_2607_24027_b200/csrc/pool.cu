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
// A thread-block cluster takes one head.  Each CTA sums its share of the keys, first for the mean, then for a
// partial C_K in registers (256 threads, 8 x 8 or 4 x 4 each); the partial sums are added through distributed
// shared memory in rank order (bit-stable run to run), every CTA gathers the whole C_K and forms Y = Qbar C_K for
// its share of the query blocks.  A share of up to 88 keys stays in shared memory between the two passes, and up to
// 88 query blocks are one step: with two CTAs per SM that is the largest `work` area there is room for, and what 40
// heads of 591 blocks give a CTA of a cluster of 7.  1.5 GFLOP at that size, 60 us; three kernels (mean on 40
// CTAs; C_K with one shared-memory operand per FMA; quadratic form) took 198 us.
constexpr int kMomentRows = 88;

template <int D>
constexpr size_t moments_smem() {                // C_K, then (in turn) keys / a reduced strip / pooled queries
  constexpr size_t work = sizeof(float) * kMomentRows * D, strip = sizeof(float) * D * D / 2;
  return sizeof(float) * D * D + (work > strip ? work : strip);
}

template <int D>
__global__ void __launch_bounds__(256, 2) thresholds_moments_kernel(WsPtrs ws, int Nq, int Nk, float scale, float beta) {
  constexpr int T = D / 16;                      // C_K rows and columns per thread (8 or 4)
  constexpr int G = 256 / D;
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  const int n_cta = (int)cluster.num_blocks(), rank = (int)cluster.block_rank();
  extern __shared__ __align__(16) float smem_f[];
  float* cov = smem_f;                           // [D][D]
  float* work = smem_f + D * D;
  __shared__ __align__(16) float part[G][D], sum_s[D], mean_s[D];
  const int bh = blockIdx.y, tid = threadIdx.x;
  const int ty = tid / 16, tx = tid % 16;
  const float* kc = ws.kc + (size_t)bh * Nk * D;
  const int per_k = ceil_div(Nk, n_cta);
  const int j_begin = min(Nk, rank * per_k), j_end = min(Nk, j_begin + per_k);

  // copies n rows of D floats to `work`
  auto stage = [&](const float* src, int n) {
#pragma unroll 4
    for (int e = tid; e < n * (D / 4); e += 256)
      reinterpret_cast<float4*>(work)[e] = reinterpret_cast<const float4*>(src)[e];
  };
  kernel_wait();
  const bool resident = j_end - j_begin <= kMomentRows;

  // ---- m_K
  {
    if (resident) {
      stage(kc + (size_t)j_begin * D, j_end - j_begin);
      __syncthreads();
    }
    const float* x = resident ? work : kc + (size_t)j_begin * D;
    const int c = tid % D, g = tid / D;
    float s = 0.f;
#pragma unroll 8
    for (int j = g; j < j_end - j_begin; j += G) s += x[(size_t)j * D + c];
    part[g][c] = s;
    __syncthreads();
    if (g == 0) {
      float r = 0.f;
#pragma unroll
      for (int y = 0; y < G; ++y) r += part[y][c];
      sum_s[c] = r;
    }
    cluster.sync();
    if (g == 0) {
      float other[8], r = 0.f;
#pragma unroll
      for (int y = 0; y < 8; ++y) other[y] = y < n_cta ? cluster.map_shared_rank(sum_s, y)[c] : 0.f;
#pragma unroll
      for (int y = 0; y < 8; ++y) r += other[y];
      mean_s[c] = r / (float)Nk;
    }
    __syncthreads();
  }

  // ---- this CTA's share of C_K.  Thread (ty, tx) owns rows and columns 4 ty + r (+ 64), 4 tx + c (+ 64).
  float2 acc[T][T / 2];
#pragma unroll
  for (int r = 0; r < T; ++r)
#pragma unroll
    for (int c = 0; c < T / 2; ++c) acc[r][c] = make_float2(0.f, 0.f);
  for (int j0 = j_begin; j0 < j_end; j0 += kMomentRows) {
    const int nj = min(kMomentRows, j_end - j0);
    if (!resident) {
      stage(kc + (size_t)j0 * D, nj);
      __syncthreads();
    }
    for (int e = tid; e < nj * (D / 4); e += 256) {
      float4 x = reinterpret_cast<float4*>(work)[e];
      const float4 m = *reinterpret_cast<const float4*>(mean_s + (e % (D / 4)) * 4);
      x.x -= m.x; x.y -= m.y; x.z -= m.z; x.w -= m.w;
      reinterpret_cast<float4*>(work)[e] = x;
    }
    __syncthreads();
#pragma unroll 2
    for (int jj = 0; jj < nj; ++jj) {
      const float* x = work + jj * D;
      float a[T], b[T];
#pragma unroll
      for (int h = 0; h < T / 4; ++h) {
        *reinterpret_cast<float4*>(a + 4 * h) = *reinterpret_cast<const float4*>(x + 64 * h + 4 * ty);
        *reinterpret_cast<float4*>(b + 4 * h) = *reinterpret_cast<const float4*>(x + 64 * h + 4 * tx);
      }
#pragma unroll
      for (int r = 0; r < T; ++r)
#pragma unroll
        for (int c = 0; c < T / 2; ++c)
          acc[r][c] = __ffma2_rn(make_float2(a[r], a[r]), make_float2(b[2 * c], b[2 * c + 1]), acc[r][c]);
    }
    __syncthreads();
  }
  const float inv = 1.f / (float)Nk;
#pragma unroll
  for (int r = 0; r < T; ++r)
#pragma unroll
    for (int h = 0; h < T / 4; ++h) {
      const float2 lo = acc[r][2 * h], hi = acc[r][2 * h + 1];
      *reinterpret_cast<float4*>(cov + (size_t)((r / 4) * 64 + 4 * ty + r % 4) * D + 64 * h + 4 * tx) =
          make_float4(lo.x * inv, lo.y * inv, hi.x * inv, hi.y * inv);
    }
  if (n_cta > 1) {
    cluster.sync();
    // add the partial matrices, one strip per CTA, then gather the strips
    constexpr int kPieces = D * D / 4;
    const int per = ceil_div(kPieces, n_cta);
    const int e0 = min(kPieces, rank * per), e1 = min(kPieces, e0 + per);
    for (int e = e0 + tid; e < e1; e += 256) {
      float4 y[8], r = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int x = 0; x < 8; ++x)
        y[x] = x < n_cta ? reinterpret_cast<const float4*>(cluster.map_shared_rank(cov, x))[e] : r;
#pragma unroll
      for (int x = 0; x < 8; ++x) { r.x += y[x].x; r.y += y[x].y; r.z += y[x].z; r.w += y[x].w; }
      reinterpret_cast<float4*>(work)[e - e0] = r;
    }
    cluster.sync();
#pragma unroll 8
    for (int e = tid; e < kPieces; e += 256)
      reinterpret_cast<float4*>(cov)[e] = reinterpret_cast<const float4*>(cluster.map_shared_rank(work, e / per))[e % per];
    cluster.sync();                              // the strips are read: `work` is free again, and a CTA may leave
  } else {
    __syncthreads();
  }

  // ---- Y = Qbar C_K and the row sums of Y o Qbar; thread (ty, tx) owns query blocks ty + 16 a and columns
  //      4 tx + c (+ 64)
  const int per_q = ceil_div(Nq, n_cta);
  const int i_begin = min(Nq, rank * per_q), i_end = min(Nq, i_begin + per_q);
  auto rows = [&](auto a_c, int i0) {
    constexpr int A = decltype(a_c)::value;
    const int nq = min(min(16 * A, kMomentRows), i_end - i0);
    stage(ws.qbar + ((size_t)bh * Nq + i0) * D, nq);
    __syncthreads();
    const float* q_row[A];                       // (rows past the last repeat it and are not stored)
#pragma unroll
    for (int a = 0; a < A; ++a) q_row[a] = work + min(ty + 16 * a, nq - 1) * D;
    float2 y[A][T / 2];
#pragma unroll
    for (int a = 0; a < A; ++a)
#pragma unroll
      for (int c = 0; c < T / 2; ++c) y[a][c] = make_float2(0.f, 0.f);
#pragma unroll 1
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
  // One cluster per head, as large as leaves every CTA an SM of its own with room for the clusters to be packed
  // into GPCs: two CTAs on an SM share its FMA pipes and take twice as long.  40 heads x 591 blocks: clusters of 2 / 3 /
  // 4 / 7 take 80 / 60 / 82 / 77 us; 24 heads x 300: 4 / 5 / 6 take 27 / 24 / 38 us.
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const int fit = sms * 17 / 20 / p.BH;
  const int n_cta = fit < 1 ? 1 : (fit > 8 ? 8 : fit);
  if (n_launches) *n_launches += 1;
  return launch_after(thresholds_moments_kernel<D>, dim3(n_cta, p.BH), 256, moments_smem<D>(), moments_smem<D>(), n_cta, stream, ws, p.Nq, p.Nk,
                      p.scale, p.beta);
}

cudaError_t launch_thresholds(const Problem& p, const WsPtrs& ws, cudaStream_t stream, int* n_launches) {
  return p.d == 128 ? thresholds_impl<128>(p, ws, stream, n_launches)
                    : thresholds_impl<64>(p, ws, stream, n_launches);
}

}  // namespace sol
