// Column normalization of R (n x r) into Q, and what the two rank-r updates after it read: one pass that takes the columns'
// sums of squares (and R's largest magnitude), one pass that writes Q and, beside it, Q as a half array for the weight
// update and R as an operand pair for the error feedback.
#pragma once
#include <cuda_fp16.h>

#include "bf16_kernels.cuh"
#include "dion_common.cuh"

namespace dion {

// Blocks of 256 threads take 128 columns x rows_per_chunk rows: a lane holds four columns (V4: neighbours, 16-byte accesses;
// else 32 apart), a warp every eighth row.  A thread per column walked its chunk's rows and, before that, all chunks'
// partial sums one dependent load after the other (16384 x 256: 296 chunks, 14 us of latency); with a warp per row both
// chains are an eighth as long.
constexpr int CN_THREADS = 256;
constexpr int CN_WARPS = CN_THREADS / 32;

template <bool V4>
__device__ __forceinline__ i64 cn_col(i64 j0, int lane, int k) { return V4 ? j0 + 4 * lane + k : j0 + lane + 32 * k; }

template <bool V4>
__device__ __forceinline__ void cn_load(const float* __restrict__ row, i64 j0, int lane, i64 r, float (&v)[4]) {
  if (V4) {
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j0 + 4 * lane < r) t = *reinterpret_cast<const float4*>(row + j0 + 4 * lane);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else {
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = (j0 + lane + 32 * k < r) ? row[j0 + lane + 32 * k] : 0.f;
  }
}

// v[k] summed over the block's warps, in the order of the warps; every thread gets its columns' sums.
__device__ __forceinline__ void cn_block_sum(float (&v)[4], float (*red)[128]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 4; ++k) red[warp][lane + 32 * k] = v[k];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < CN_WARPS; ++w) s += red[w][lane + 32 * k];
    v[k] = s;
  }
}

// The chunks' partial sums of the thread's columns, added up (always in this order: the sharded form hands the sums out).
template <bool V4>
__device__ __forceinline__ void cn_sum_chunks(const float* __restrict__ part, int chunks, i64 j0, i64 r, float (*red)[128], float (&s)[4]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool aligned = ((uintptr_t)part & 15) == 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) s[k] = 0.f;
#pragma unroll 4
  for (int c = warp; c < chunks; c += CN_WARPS) {
    float v[4];
    if (!V4 || aligned) {
      cn_load<V4>(part + (i64)c * r, j0, lane, r, v);
    } else {      // (a caller's array of sums may lie anywhere)
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = j0 + 4 * lane < r ? part[(i64)c * r + j0 + 4 * lane + k] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] += v[k];
  }
  cn_block_sum(s, red);
}

// part[chunk][j] = sum over the chunk's rows of R[i][j]^2; grid = (ceil(r / 128), chunks, matrices of a chain: R, part and amax
// wstride floats apart, skip flags a state slot apart).  amax (optional): the blocks' largest |R|, gridDim.x * gridDim.y of them.
template <bool V4>
__global__ void __launch_bounds__(CN_THREADS) k_colsumsq_partial(const float* __restrict__ R, i64 ld, i64 n, i64 r, i64 rows_per_chunk,
                                                                 float* __restrict__ part, float* __restrict__ amax,
                                                                 const int* __restrict__ skip_flag, i64 wstride) {
  pdl_enter();
  if (skip_flag != nullptr && skip_flag[(i64)blockIdx.z * OS_SLOT_INTS] != 0) return;
  __shared__ float red[CN_WARPS][128];
  __shared__ float redm[CN_WARPS];
  R += (i64)blockIdx.z * wstride; part += (i64)blockIdx.z * wstride;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const i64 j0 = (i64)blockIdx.x * 128;
  const i64 i0 = (i64)blockIdx.y * rows_per_chunk, i1 = min(n, i0 + rows_per_chunk);
  float s[4] = {0.f, 0.f, 0.f, 0.f}, m = 0.f;
#pragma unroll 4
  for (i64 i = i0 + warp; i < i1; i += CN_WARPS) {
    float v[4];
    cn_load<V4>(R + i * ld, j0, lane, r, v);
#pragma unroll
    for (int k = 0; k < 4; ++k) { s[k] = fmaf(v[k], v[k], s[k]); m = fmaxf(m, fabsf(v[k])); }
  }
  if (amax != nullptr) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) redm[warp] = m;
  }
  cn_block_sum(s, red);
  if (warp == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const i64 j = cn_col<V4>(j0, lane, k);
      if (j < r) part[(i64)blockIdx.y * r + j] = s[k];
    }
    if (amax != nullptr && lane == 0) {
      float t = redm[0];
#pragma unroll
      for (int w = 1; w < CN_WARPS; ++w) t = fmaxf(t, redm[w]);
      amax[(i64)blockIdx.z * wstride + (i64)blockIdx.y * gridDim.x + blockIdx.x] = t;
    }
  }
}

// out[j] = the chunks' partial sums added up: the squared column norms of a shard's rows, handed to the caller for the
// all-reduce over the shards (1D-sharded Dion).
template <bool V4>
__global__ void __launch_bounds__(CN_THREADS) k_colsumsq_finish(const float* __restrict__ part, int chunks, i64 r, float* __restrict__ out,
                                                                const int* __restrict__ skip_flag) {
  pdl_enter();
  if (skip_flag != nullptr && *skip_flag != 0) return;
  __shared__ float red[CN_WARPS][128];
  const i64 j0 = (i64)blockIdx.x * 128;
  float s[4];
  cn_sum_chunks<V4>(part, chunks, j0, r, red, s);
  if (threadIdx.x < 32) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const i64 j = cn_col<V4>(j0, threadIdx.x, k);
      if (j < r) out[j] = s[k];
    }
  }
}

// What k_colnorm_apply writes beside Q (all optional; r a multiple of 8 then), per matrix of a chain in the scratch slices.
struct ColnormPairs {
  int kind;                // 0: nothing, else what R becomes: CN_HALF or CN_BF16, a pair; CN_ONE, a bf16 array
  void* qh; float qscale;  // Q as a half array, scaled (CN_ONE: as a bf16 array) ...
  int qpair;               // ... and what that leaves of it, n * r elements behind
  void* hi;                // R's array or pair: hi, then lo n * r elements behind it
  const float* amax; int nmax;   // CN_HALF: R's block maxima; its scale puts the largest magnitude in [2^13, 2^14)
  float* scal;             // ... and the factor that takes the scales out of the product with U's pair,
  const float* other;      // or with another pair (optional: its 1 / scale)
  int* os;                 // CN_HALF, optional: state slots; the pair of a matrix whose OS_WIDE is set is a bf16 pair.  With
  const float* range;      // `range` the flag is set here: ranges (k_range_partial) of R and, behind them, of U, of
  int nrange;              // this many blocks.  With qpair (Lazy-Dion) the flag is OS_P32 instead: U goes to qh as it is, in fp32,
                           // and OS_USE32 and OS_USEHALF are set for the updates (both when the step is cancelled)
};
enum : int { CN_HALF = 1, CN_BF16 = 2, CN_ONE = 3 };

// d_j = sqrt(sum of the partials); Q[i][j] = R[i][j] / (d_j + eps).  Grid as for k_colsumsq_partial with row blocks of its own
// (every block adds the chunks' sums up again, so a chain of many matrices takes fewer and larger ones: 48 of 768 x 192 in
// blocks of 32 rows 47 us, 27 us now); the blocks of row block 0 also export d.  Q and d_out come from pointer tables; qvec: Q's rows are 16-byte aligned.
// QP: Q's half array is a pair (x.qpair).
template <bool V4, bool QP>
__global__ void __launch_bounds__(CN_THREADS, 3) k_colnorm_apply(const float* __restrict__ R, i64 ldr, i64 n, i64 r, i64 rows_per_chunk, int chunks,
                                                              const float* __restrict__ part, float eps, const ChainPtrs Qs, i64 ldq, int qvec,
                                                              float* __restrict__ d_ws, const ChainPtrs ds, int* __restrict__ status,
                                                              const int* __restrict__ skip_flag, i64 wstride, ColnormPairs x,
                                                              int* __restrict__ skipped) {
  pdl_enter();
  const i64 b = blockIdx.z;
  if (skip_flag != nullptr && skip_flag[b * OS_SLOT_INTS] != 0) {
    if (threadIdx.x == 0 && blockIdx.x == 0 && blockIdx.y == 0) {
      atomicAdd(skipped, 1);      // (once per step: the count of cancelled steps)
      if (QP && x.os != nullptr) x.os[b * OS_SLOT_INTS + OS_USE32] = x.os[b * OS_SLOT_INTS + OS_USEHALF] = 1;
    }
    return;
  }
  __shared__ float red[CN_WARPS][128];
  __shared__ float redm[CN_WARPS];
  R += b * wstride; part += b * wstride; d_ws += b * wstride;
  float* __restrict__ Q = reinterpret_cast<float*>(const_cast<void*>(Qs.p[b]));
  float* __restrict__ d_out = reinterpret_cast<float*>(const_cast<void*>(ds.p[b]));
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const i64 j0 = (i64)blockIdx.x * 128;
  float m = 0.f;
  if (x.kind == CN_HALF) {
    const float* a = x.amax + b * wstride;
    for (int e = threadIdx.x; e < x.nmax; e += CN_THREADS) m = fmaxf(m, a[e]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) redm[warp] = m;
  }
  float s[4];
  cn_sum_chunks<V4>(part, chunks, j0, r, red, s);      // (its barrier also covers redm)
  float rscale = 1.f;
  bool bf16 = x.kind == CN_BF16;
  if (x.kind == CN_HALF) {
    m = redm[0];
#pragma unroll
    for (int w = 1; w < CN_WARPS; ++w) m = fmaxf(m, redm[w]);
    if (x.range != nullptr) {      // (U's scale is 2^13, its entries are at most 1)
      float mw, nw, mu, nu;
      range_of_blocks(x.range, x.nrange, mw, nw);
      range_of_blocks(x.range + 2 * x.nrange, x.nrange, mu, nu);
      m = mw;
      bf16 = range_is_wide(mw, nw, RANGE_UPDATE) || nu < RANGE_UPDATE;
      if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) x.os[OS_WIDE] = bf16 ? 1 : 0;
    } else if (!QP && x.os != nullptr) {
      bf16 = x.os[b * OS_SLOT_INTS + OS_WIDE] != 0;
    }
    const int e = f16_scale_exponent(m);
    rscale = ldexpf(1.f, e);
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0)
      x.scal[b * wstride] = bf16 ? 1.f : x.other != nullptr ? ldexpf(1.f, -e) * x.other[b * wstride] : ldexpf(1.f, -e - HS_U_BITS);
  }
  bool use32 = false;
  if (QP && x.os != nullptr) {
    int* os = x.os + b * OS_SLOT_INTS;
    use32 = os[OS_P32] != 0;
    if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) { os[OS_USE32] = use32 ? 1 : 0; os[OS_USEHALF] = use32 ? 0 : 1; }
  }
  float inv[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float d = sqrtf(s[k]);
    const i64 j = cn_col<V4>(j0, lane, k);
    if (blockIdx.y == 0 && warp == 0 && j < r) {
      d_ws[j] = d;
      if (d_out != nullptr) d_out[j] = d;
      if (!isfinite(d)) atomicOr(status, DION_STATUS_NONFINITE);
    }
    inv[k] = 1.f / (d + eps);
  }
  const i64 i0 = (i64)blockIdx.y * rows_per_chunk, i1 = min(n, i0 + rows_per_chunk);
  for (i64 ib = i0 + warp; ib < i1; ib += 4 * CN_WARPS) {
  float rows[4][4];      // four rows in flight (the stores below would keep the compiler from overlapping them)
#pragma unroll
  for (int t = 0; t < 4; ++t)
    if (ib + t * CN_WARPS < i1) cn_load<V4>(R + (ib + t * CN_WARPS) * ldr, j0, lane, r, rows[t]);
#pragma unroll
  for (int t = 0; t < 4; ++t) {
    const i64 i = ib + t * CN_WARPS;
    if (i >= i1) break;
    const float (&v)[4] = rows[t];
    const float q[4] = {v[0] * inv[0], v[1] * inv[1], v[2] * inv[2], v[3] * inv[3]};
    if (V4) {
      const i64 j = j0 + 4 * lane;
      if (j >= r) continue;
      if (Q == nullptr) {      // (only its half arrays are wanted)
      } else if (qvec) {
        *reinterpret_cast<float4*>(Q + i * ldq + j) = make_float4(q[0], q[1], q[2], q[3]);
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) Q[i * ldq + j + k] = q[k];
      }
      if (QP && use32) {
        *reinterpret_cast<float4*>(reinterpret_cast<float*>(x.qh) + b * wstride + i * r + j) = make_float4(q[0], q[1], q[2], q[3]);
      } else if (x.kind != 0) {
        const i64 at = 2 * b * wstride + i * r + j;
        __half h[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) h[k] = __float2half_rn(x.qscale * q[k]);
        uint2 q16 = *reinterpret_cast<const uint2*>(h), hi, lo;
        if (x.kind == CN_HALF && !bf16) {
          __half l[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float t = rscale * v[k];
            h[k] = __float2half_rn(t);
            l[k] = __float2half_rn(t - __half2float(h[k]));
          }
          hi = *reinterpret_cast<const uint2*>(h); lo = *reinterpret_cast<const uint2*>(l);
        } else {
          float t[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) t[k] = __bfloat162float(__float2bfloat16_rn(v[k]));
          hi.x = pack_bf16x2(t[0], t[1]); hi.y = pack_bf16x2(t[2], t[3]);
          lo.x = pack_bf16x2(v[0] - t[0], v[1] - t[1]); lo.y = pack_bf16x2(v[2] - t[2], v[3] - t[3]);
          if (x.kind == CN_ONE) { q16.x = pack_bf16x2(q[0], q[1]); q16.y = pack_bf16x2(q[2], q[3]); }
        }
        *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(x.qh) + at) = q16;
        if constexpr (QP) {
          const __half* qh = reinterpret_cast<const __half*>(&q16);
          __half l[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) l[k] = __float2half_rn(x.qscale * q[k] - __half2float(qh[k]));
          *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(x.qh) + at + n * r) = *reinterpret_cast<const uint2*>(l);
        }
        *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(x.hi) + at) = hi;
        if (x.kind != CN_ONE) *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(x.hi) + at + n * r) = lo;
      }
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const i64 j = j0 + lane + 32 * k;
        if (j < r) Q[i * ldq + j] = q[k];
      }
    }
  }
  }
}

}  // namespace dion
