// Operand preparation in scratch: bf16(M + G) and bf16 copies (bf16-operand mode), M + G in fp32, and
// TF32-rounded copies of the factors of the weight update (fp32 mode).
#pragma once

#include <cuda_fp16.h>

#include "dion_common.cuh"

namespace dion {

// The first kernel of a step clears the state slots of the chain's matrices (blockIdx.y; a memset of its own was 2 us).
__device__ __forceinline__ void clear_slot(int* slots) {
  if (slots != nullptr && blockIdx.x == 0 && threadIdx.x < OS_SLOT_INTS) slots[blockIdx.y * OS_SLOT_INTS + threadIdx.x] = 0;
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// B16 = bf16(M + G), rows x cols, B16 dense with leading dimension cols (a multiple of 8).
// One thread per 8 consecutive elements of a row.  VEC: M (and G) rows start 16-byte
// aligned (pointer and leading dimension), so the loads are 128-bit.
template <bool VEC>
__global__ void __launch_bounds__(256) k_form_b16(const float* __restrict__ M, i64 ldm, const void* __restrict__ G,
                                                  i64 ldg, int g_mode, i64 rows, i64 cols,
                                                  __nv_bfloat16* __restrict__ out, int* __restrict__ slots) {
  pdl_enter();
  clear_slot(slots);
  const i64 per_row = cols / 8;
  const i64 total = rows * per_row;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    const i64 i = row_of(e, per_row), c = (e - i * per_row) * 8;
    float v[8];
    const float* mp = M + i * ldm + c;
    if (VEC) {
      const float4 a = __ldg(reinterpret_cast<const float4*>(mp)), b = __ldg(reinterpret_cast<const float4*>(mp) + 1);
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = mp[q];
    }
    if (g_mode == ADD_F32) {
      const float* gp = reinterpret_cast<const float*>(G) + i * ldg + c;
      if (VEC) {
        const float4 a = __ldg(reinterpret_cast<const float4*>(gp)), b = __ldg(reinterpret_cast<const float4*>(gp) + 1);
        v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w; v[4] += b.x; v[5] += b.y; v[6] += b.z; v[7] += b.w;
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] += gp[q];
      }
    } else if (g_mode == ADD_BF16) {
      const __nv_bfloat16* gp = reinterpret_cast<const __nv_bfloat16*>(G) + i * ldg + c;
      if (VEC) {
        const uint4 w = __ldg(reinterpret_cast<const uint4*>(gp));
        const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(&ww[q]);
          v[2 * q] += __low2float(h); v[2 * q + 1] += __high2float(h);
        }
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] += __bfloat162float(gp[q]);
      }
    }
    uint4 o;
    o.x = pack_bf16x2(v[0], v[1]); o.y = pack_bf16x2(v[2], v[3]);
    o.z = pack_bf16x2(v[4], v[5]); o.w = pack_bf16x2(v[6], v[7]);
    *reinterpret_cast<uint4*>(out + i * cols + c) = o;
  }
}

// B32 = M + G in fp32, rows x cols (cols a multiple of 4), B32 dense with leading dimension cols: the sum the
// fused operand formation of the contraction kernel computes, formed once per step where two products and the
// error feedback read it.  One thread per 4 consecutive elements of a row; VEC as above.
// hi / lo (optional, both or neither; cols a multiple of 8 then): the same sum as a pair of bf16 arrays, hi = bf16(sum),
// lo = bf16(sum - hi), dense like out: the operand of the products that run on bf16 pairs.
constexpr int FORM_BATCH = 4;
template <bool VEC>
__device__ __forceinline__ void form_b32_body(const float* __restrict__ M, i64 ldm, const void* __restrict__ G,
                                              i64 ldg, int g_mode, i64 rows, i64 cols, float* __restrict__ out,
                                              __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo) {
  const i64 per_row = cols / 4;
  const i64 total = rows * per_row;
  // (FORM_BATCH pieces in flight per thread: the sums' stores would keep the compiler from overlapping the loads)
  const i64 stride = (i64)gridDim.x * blockDim.x;
  for (i64 e0 = (i64)blockIdx.x * blockDim.x + threadIdx.x; e0 < total; e0 += FORM_BATCH * stride) {
   float4 mv[FORM_BATCH], gv[FORM_BATCH];
   i64 at[FORM_BATCH];
#pragma unroll
   for (int u = 0; u < FORM_BATCH; ++u) {
    const i64 e = e0 + u * stride;
    if (e >= total) break;
    const i64 i = row_of(e, per_row), c = (e - i * per_row) * 4;
    at[u] = i * cols + c;
    const float* mp = M + i * ldm + c;
    if (VEC) mv[u] = __ldg(reinterpret_cast<const float4*>(mp));
    else mv[u] = make_float4(mp[0], mp[1], mp[2], mp[3]);
    if (g_mode == ADD_F32) {
      const float* gp = reinterpret_cast<const float*>(G) + i * ldg + c;
      if (VEC) gv[u] = __ldg(reinterpret_cast<const float4*>(gp));
      else gv[u] = make_float4(gp[0], gp[1], gp[2], gp[3]);
    } else if (g_mode == ADD_BF16) {
      const __nv_bfloat16* gp = reinterpret_cast<const __nv_bfloat16*>(G) + i * ldg + c;
      if (VEC) {
        const uint2 w = __ldg(reinterpret_cast<const uint2*>(gp));
        gv[u].x = __uint_as_float(w.x); gv[u].y = __uint_as_float(w.y);
      } else {
        gv[u] = make_float4(__bfloat162float(gp[0]), __bfloat162float(gp[1]), __bfloat162float(gp[2]), __bfloat162float(gp[3]));
      }
    }
   }
#pragma unroll
   for (int u = 0; u < FORM_BATCH; ++u) {
    if (e0 + u * stride >= total) break;
    float4 v = mv[u], g = gv[u];
    if (VEC && g_mode == ADD_BF16) {      // (still the four bf16 values)
      const uint32_t w0 = __float_as_uint(g.x), w1 = __float_as_uint(g.y);
      const __nv_bfloat162 lo2 = *reinterpret_cast<const __nv_bfloat162*>(&w0);
      const __nv_bfloat162 hi2 = *reinterpret_cast<const __nv_bfloat162*>(&w1);
      g = make_float4(__low2float(lo2), __high2float(lo2), __low2float(hi2), __high2float(hi2));
    }
    if (g_mode != ADD_NONE) { v.x += g.x; v.y += g.y; v.z += g.z; v.w += g.w; }
    *reinterpret_cast<float4*>(out + at[u]) = v;
    if (hi != nullptr) {
      const float h0 = __bfloat162float(__float2bfloat16_rn(v.x)), h1 = __bfloat162float(__float2bfloat16_rn(v.y));
      const float h2 = __bfloat162float(__float2bfloat16_rn(v.z)), h3 = __bfloat162float(__float2bfloat16_rn(v.w));
      uint2 oh, ol;
      oh.x = pack_bf16x2(h0, h1); oh.y = pack_bf16x2(h2, h3);
      ol.x = pack_bf16x2(v.x - h0, v.y - h1); ol.y = pack_bf16x2(v.z - h2, v.w - h3);
      *reinterpret_cast<uint2*>(hi + at[u]) = oh;
      *reinterpret_cast<uint2*>(lo + at[u]) = ol;
    }
   }
  }
}
template <bool VEC>
__global__ void __launch_bounds__(256, 3) k_form_b32(const float* __restrict__ M, i64 ldm, const void* __restrict__ G,
                                                  i64 ldg, int g_mode, i64 rows, i64 cols, float* __restrict__ out,
                                                  __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo, int* __restrict__ slots) {
  pdl_enter();
  clear_slot(slots);
  form_b32_body<VEC>(M, ldm, G, ldg, g_mode, rows, cols, out, hi, lo);
}
// The same for every matrix of a chain in one launch (blockIdx.y): the caller's M and G from pointer tables, the
// outputs in the scratch slices, `ostride` floats apart.
template <bool VEC>
__global__ void __launch_bounds__(256, 3) k_form_b32_chain(const ChainPtrs Ms, i64 ldm, const ChainPtrs Gs, i64 ldg, int g_mode,
                                                        i64 rows, i64 cols, float* __restrict__ out,
                                                        __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo,
                                                        i64 ostride, int* __restrict__ slots) {
  pdl_enter();
  clear_slot(slots);
  const i64 b = blockIdx.y;
  form_b32_body<VEC>(reinterpret_cast<const float*>(Ms.p[b]), ldm, Gs.p[b], ldg, g_mode, rows, cols, out + b * ostride,
                     hi != nullptr ? hi + 2 * b * ostride : nullptr, lo != nullptr ? lo + 2 * b * ostride : nullptr);
}

// out = bf16(src), rows x cols (cols a multiple of 8, src rows 16-byte aligned), out dense.
// skip_flag (optional): nothing is written when *skip_flag != 0.
__global__ void __launch_bounds__(256) k_to_bf16(const float* __restrict__ src, i64 lds, i64 rows, i64 cols,
                                                 __nv_bfloat16* __restrict__ out, const int* __restrict__ skip_flag) {
  pdl_enter();
  if (skip_flag != nullptr && *skip_flag != 0) return;
  const i64 per_row = cols / 8;
  const i64 total = rows * per_row;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    const i64 i = row_of(e, per_row), c = (e - i * per_row) * 8;
    const float4 a = *reinterpret_cast<const float4*>(src + i * lds + c);
    const float4 b = *(reinterpret_cast<const float4*>(src + i * lds + c) + 1);
    uint4 o;
    o.x = pack_bf16x2(a.x, a.y); o.y = pack_bf16x2(a.z, a.w);
    o.z = pack_bf16x2(b.x, b.y); o.w = pack_bf16x2(b.z, b.w);
    *reinterpret_cast<uint4*>(out + i * cols + c) = o;
  }
}

// hi = bf16(src), lo = bf16(src - hi): src ~ hi + lo to 16 significant bits.  rows x cols (cols a multiple of 8,
// src rows 16-byte aligned), hi and lo dense.  skip_flag (optional): nothing is written when *skip_flag != 0.
// copy (optional): src also as a dense fp32 array; one (optional): half(one_scale src), dense (k_round_f16's values)
__device__ __forceinline__ void split_bf16_body(const float* __restrict__ src, i64 lds, i64 rows, i64 cols,
                                                __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo,
                                                float* __restrict__ copy, __half* __restrict__ one, float one_scale) {
  const i64 per_row = cols / 8;
  const i64 total = rows * per_row;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    const i64 i = row_of(e, per_row), c = (e - i * per_row) * 8;
    const float4 a = *reinterpret_cast<const float4*>(src + i * lds + c);
    const float4 b = *(reinterpret_cast<const float4*>(src + i * lds + c) + 1);
    const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    float h[8], l[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      h[q] = __bfloat162float(__float2bfloat16_rn(v[q]));
      l[q] = v[q] - h[q];
    }
    uint4 oh, ol;
    oh.x = pack_bf16x2(h[0], h[1]); oh.y = pack_bf16x2(h[2], h[3]); oh.z = pack_bf16x2(h[4], h[5]); oh.w = pack_bf16x2(h[6], h[7]);
    ol.x = pack_bf16x2(l[0], l[1]); ol.y = pack_bf16x2(l[2], l[3]); ol.z = pack_bf16x2(l[4], l[5]); ol.w = pack_bf16x2(l[6], l[7]);
    *reinterpret_cast<uint4*>(hi + i * cols + c) = oh;
    *reinterpret_cast<uint4*>(lo + i * cols + c) = ol;
    if (copy != nullptr) {
      *reinterpret_cast<float4*>(copy + i * cols + c) = a;
      *(reinterpret_cast<float4*>(copy + i * cols + c) + 1) = b;
    }
    if (one != nullptr) {
      __half t[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) t[q] = __float2half_rn(one_scale * v[q]);
      *reinterpret_cast<uint4*>(one + i * cols + c) = *reinterpret_cast<const uint4*>(t);
    }
  }
}
__global__ void __launch_bounds__(256) k_split_bf16(const float* __restrict__ src, i64 lds, i64 rows, i64 cols,
                                                    __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo,
                                                    const int* __restrict__ skip_flag, __half* __restrict__ one, float one_scale) {
  pdl_enter();
  if (skip_flag != nullptr && *skip_flag != 0) return;
  split_bf16_body(src, lds, rows, cols, hi, lo, nullptr, one, one_scale);
}
// One launch over the matrices of a chain (blockIdx.y): sources from a pointer table, outputs `ostride` floats
// apart in the scratch slices, skip flags `skip_stride` ints apart.
__global__ void __launch_bounds__(256) k_split_bf16_chain(const ChainPtrs srcs, i64 lds, i64 rows, i64 cols,
                                                          __nv_bfloat16* __restrict__ hi, __nv_bfloat16* __restrict__ lo,
                                                          i64 ostride, const int* __restrict__ skip_flag, i64 skip_stride,
                                                          float* __restrict__ copy, __half* __restrict__ one, float one_scale) {
  pdl_enter();
  const i64 b = blockIdx.y;
  if (skip_flag != nullptr && skip_flag[b * skip_stride] != 0) return;
  split_bf16_body(reinterpret_cast<const float*>(srcs.p[b]), lds, rows, cols, hi + 2 * b * ostride, lo + 2 * b * ostride,
                  copy != nullptr ? copy + b * ostride : nullptr, one != nullptr ? one + 2 * b * ostride : nullptr, one_scale);
}

// Dense fp32 copies of a chain's matrices (blockIdx.y; sources from a pointer table, 16-byte aligned rows, cols a multiple
// of 4), `ostride` floats apart.
__global__ void __launch_bounds__(256) k_copy_chain(const ChainPtrs srcs, i64 lds, i64 rows, i64 cols, float* __restrict__ out, i64 ostride) {
  pdl_enter();
  const float* __restrict__ src = reinterpret_cast<const float*>(srcs.p[blockIdx.y]);
  out += (i64)blockIdx.y * ostride;
  const i64 per_row = cols / 4, total = rows * per_row;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    const i64 i = row_of(e, per_row), c = (e - i * per_row) * 4;
    *reinterpret_cast<float4*>(out + i * cols + c) = *reinterpret_cast<const float4*>(src + i * lds + c);
  }
}

// out = src with every value rounded to the nearest TF32 number (10 explicit mantissa bits, ties away
// from zero), rows x cols (cols a multiple of 4, src rows 16-byte aligned), out dense.  The tensor core
// truncates an fp32 operand to TF32 when it reads it; on pre-rounded values that truncation is exact, so a
// single-pass TF32 product of such arrays carries an unbiased operand error of at most 2^-11 relative.
// skip_flag (optional): nothing is written when *skip_flag != 0.
__device__ __forceinline__ void round_tf32_body(const float* __restrict__ src, i64 lds, i64 rows, i64 cols,
                                                float* __restrict__ out) {
  const i64 per_row = cols / 4;
  const i64 total = rows * per_row;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    const i64 i = row_of(e, per_row), c = (e - i * per_row) * 4;
    const float4 a = *reinterpret_cast<const float4*>(src + i * lds + c);
    uint4 o;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(o.x) : "f"(a.x));
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(o.y) : "f"(a.y));
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(o.z) : "f"(a.z));
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(o.w) : "f"(a.w));
    *reinterpret_cast<uint4*>(out + i * cols + c) = o;
  }
}
__global__ void __launch_bounds__(256) k_round_tf32(const float* __restrict__ src, i64 lds, i64 rows, i64 cols,
                                                    float* __restrict__ out, const int* __restrict__ skip_flag) {
  pdl_enter();
  if (skip_flag != nullptr && *skip_flag != 0) return;
  round_tf32_body(src, lds, rows, cols, out);
}
__global__ void __launch_bounds__(256) k_round_tf32_chain(const ChainPtrs srcs, i64 lds, i64 rows, i64 cols,
                                                          float* __restrict__ out, i64 ostride,
                                                          const int* __restrict__ skip_flag, i64 skip_stride) {
  pdl_enter();
  const i64 b = blockIdx.y;
  if (skip_flag != nullptr && skip_flag[b * skip_stride] != 0) return;
  round_tf32_body(reinterpret_cast<const float*>(srcs.p[b]), lds, rows, cols, out + b * ostride);
}

// out = half(scale * src), round to nearest: the factors of the weight update as IEEE half arrays (11 significant
// bits, like TF32, at the 16-bit MMA rate and half the operand bytes).  `scale` is a power of two chosen by the caller
// so that entries of a matrix with unit-norm columns sit around 1: far from half's subnormals, and at most
// sqrt(2 rows) < 65504.  rows x cols (cols a multiple of 8, src rows 16-byte aligned), out dense.
__device__ __forceinline__ void round_f16_body(const float* __restrict__ src, i64 lds, i64 rows, i64 cols, float scale,
                                               __half* __restrict__ out) {
  const i64 per_row = cols / 8;
  const i64 total = rows * per_row;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    const i64 i = row_of(e, per_row), c = (e - i * per_row) * 8;
    const float4 a = *reinterpret_cast<const float4*>(src + i * lds + c);
    const float4 b = *(reinterpret_cast<const float4*>(src + i * lds + c) + 1);
    __half2 h0 = __floats2half2_rn(scale * a.x, scale * a.y), h1 = __floats2half2_rn(scale * a.z, scale * a.w);
    __half2 h2 = __floats2half2_rn(scale * b.x, scale * b.y), h3 = __floats2half2_rn(scale * b.z, scale * b.w);
    uint4 o;
    o.x = *reinterpret_cast<uint32_t*>(&h0); o.y = *reinterpret_cast<uint32_t*>(&h1);
    o.z = *reinterpret_cast<uint32_t*>(&h2); o.w = *reinterpret_cast<uint32_t*>(&h3);
    *reinterpret_cast<uint4*>(out + i * cols + c) = o;
  }
}
__global__ void __launch_bounds__(256) k_round_f16(const float* __restrict__ src, i64 lds, i64 rows, i64 cols, float scale,
                                                   __half* __restrict__ out, const int* __restrict__ skip_flag) {
  pdl_enter();
  if (skip_flag != nullptr && *skip_flag != 0) return;
  round_f16_body(src, lds, rows, cols, scale, out);
}
// (one launch over a chain: blockIdx.y, outputs `ostride` floats apart)
__global__ void __launch_bounds__(256) k_round_f16_chain(const ChainPtrs srcs, i64 lds, i64 rows, i64 cols, float scale,
                                                         __half* __restrict__ out, i64 ostride,
                                                         const int* __restrict__ skip_flag, i64 skip_stride) {
  pdl_enter();
  const i64 b = blockIdx.y;
  if (skip_flag != nullptr && skip_flag[b * skip_stride] != 0) return;
  round_f16_body(reinterpret_cast<const float*>(srcs.p[b]), lds, rows, cols, scale, out + 2 * b * ostride);
}

// ---- a panel as a pair of IEEE half arrays, scaled: 22 significant bits at the 16-bit MMA rate ----------------
// Half has 5 exponent bits, so the panel is scaled by a power of two that puts its largest entry in [2^13, 2^14):
// entries down to 2^-17 of the largest keep all 22 bits of the pair, smaller ones an absolute error of 2^-39 of
// the largest.  Two launches: per-block maxima of |x|, then the split (every block reduces the maxima again, in
// a fixed order; block 0 also writes 1 / scale^2, the factor that takes a Gram matrix of the pair back).
// blockIdx.y: the matrix of a chain (arrays `wstride` floats apart); skip flags a state slot apart.
constexpr int AMAX_PARTS = 512;
__device__ __forceinline__ void block_max(float m, float* __restrict__ out) {      // 256 threads; out[blockIdx.x]
  __shared__ float red[256];
  red[threadIdx.x] = m;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] = fmaxf(red[threadIdx.x], red[threadIdx.x + w]);
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = red[0];
}
// The exponent of the power of two that puts amax in [2^13, 2^14): amax = f 2^ex with f in [0.5, 1) gives 14 - ex.
__device__ __forceinline__ int f16_scale_exponent(float amax) {
  int ex = 14;
  if (amax > 0.f && amax < 3.0e38f) frexpf(amax, &ex);
  return 14 - (ex < -80 ? -80 : ex);
}
// ---- the range of an array ------------------------------------------------------------------------------------
// The bits of a half pair are relative to the largest entry of its array: entries keep 22 of them down to 2^-17 of it, 17 at
// 2^-22, 6 at 2^-33, while the three-term TF32 split (22 bits) and a bf16 pair (17) keep theirs at any magnitude.  So the pass
// that finds the largest entry also looks for small ones that count: the largest entry of every piece, 128 neighbours of a row
// or 8 of a column, and the smallest of those (pieces of zeros apart).  An array with a piece below 2^-18 of its largest
// entry takes the 3xTF32 product where 22 bits are asked for (P), one with a piece below 2^-20 bf16 pairs instead of half pairs.
// (A piece that large holds an entry near its rms for any spread of values but a difference of rows, columns or blocks:
// Gaussian entries stay above 2^-8.)  512 x 768, r = 128, the lower rows 2^-24 of the upper ones: those of M off by 2.3e-5 on
// half pairs throughout, 3.4e-7 now.
constexpr int RANGE_ROWS = 8;
constexpr float RANGE_P = 3.814697265625e-06f;        // 2^-18: 20 bits and more, below the error of the sums
constexpr float RANGE_UPDATE = 9.5367431640625e-07f;  // 2^-20: as many as a bf16 pair
struct Range {
  float mx = 0.f;                  // largest magnitude
  unsigned mn = 0x7f800000u;       // smallest of the pieces' largest (float bits: ordered like the values, none is negative)
};
__device__ __forceinline__ bool range_is_wide(float mx, float mn, float limit) {      // (also: beyond what the scale can bring back)
  return mx > 0.f && (mn < mx * limit || mx < 8.3e-25f || !(mx < 3.0e38f));
}
// a lane's four entries of one row of a warp's piece (zeros where there are none); cm: its columns' largest so far
__device__ __forceinline__ void range_row(Range& g, float4 v, float (&cm)[4]) {
  const float a[4] = {fabsf(v.x), fabsf(v.y), fabsf(v.z), fabsf(v.w)};
#pragma unroll
  for (int k = 0; k < 4; ++k) cm[k] = fmaxf(cm[k], a[k]);
  const float m = fmaxf(fmaxf(a[0], a[1]), fmaxf(a[2], a[3]));
  g.mx = fmaxf(g.mx, m);
  const unsigned u = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
  if (u != 0u) g.mn = min(g.mn, u);
}
__device__ __forceinline__ void range_cols(Range& g, const float (&cm)[4]) {
#pragma unroll
  for (int k = 0; k < 4; ++k) if (cm[k] > 0.f) g.mn = min(g.mn, __float_as_uint(cm[k]));
}
// the range of rows x cols (cols a multiple of 4), a warp per 8 x 128 piece; warp w of nw
__device__ __forceinline__ void range_scan(Range& g, const float* __restrict__ src, i64 ld, i64 rows, i64 cols, bool vec, i64 w, i64 nw) {
  const i64 nct = (cols + 127) / 128, pieces = (rows + RANGE_ROWS - 1) / RANGE_ROWS * nct;
  const int lane = threadIdx.x & 31;
  for (; w < pieces; w += nw) {
    const i64 tr = row_of(w, nct), c = (w - tr * nct) * 128 + 4 * lane;
    float cm[4] = {0.f, 0.f, 0.f, 0.f};
    float4 v[RANGE_ROWS];
#pragma unroll
    for (int q = 0; q < RANGE_ROWS; ++q) {
      const i64 i = tr * RANGE_ROWS + q;
      const float* p = src + i * ld + c;
      v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i < rows && c < cols) v[q] = vec ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
    }
#pragma unroll
    for (int q = 0; q < RANGE_ROWS; ++q) range_row(g, v[q], cm);
    range_cols(g, cm);
  }
}
// 256 threads: out[blockIdx.x] and out[gridDim.x + blockIdx.x]
__device__ __forceinline__ void block_range(const Range& g, float* __restrict__ out) {
  __shared__ unsigned red[2][8];
  const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(g.mx)), n = __reduce_min_sync(0xffffffffu, g.mn);
  if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = m; red[1][threadIdx.x >> 5] = n; }
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned x = red[0][0], y = red[1][0];
#pragma unroll
    for (int w = 1; w < 8; ++w) { x = max(x, red[0][w]); y = min(y, red[1][w]); }
    out[blockIdx.x] = __uint_as_float(x); out[gridDim.x + blockIdx.x] = __uint_as_float(y);
  }
  __syncthreads();
}
// ... and over the blocks: every thread of 256 gets largest and smallest of n values each, at part and part + n.
__device__ __forceinline__ void range_of_blocks(const float* __restrict__ part, int n, float& mx, float& mn) {
  __shared__ unsigned red[2][8];
  unsigned a = 0u, b = 0x7f800000u;
  for (int e = threadIdx.x; e < n; e += 256) { a = max(a, __float_as_uint(part[e])); b = min(b, __float_as_uint(part[n + e])); }
  a = __reduce_max_sync(0xffffffffu, a); b = __reduce_min_sync(0xffffffffu, b);
  if ((threadIdx.x & 31) == 0) { red[0][threadIdx.x >> 5] = a; red[1][threadIdx.x >> 5] = b; }
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) { a = max(a, red[0][w]); b = min(b, red[1][w]); }
  mx = __uint_as_float(a); mn = __uint_as_float(b);
  __syncthreads();
}
// The ranges of arrays from a table (blockIdx.y; 16-byte aligned rows), of rows0 or, from the second on, rows1 rows: gridDim.x
// blocks' partial results `stride` floats apart.
__global__ void __launch_bounds__(256) k_range_partial(const ChainPtrs srcs, i64 ld, i64 rows0, i64 rows1, i64 cols, float* __restrict__ part,
                                                       i64 stride, const int* __restrict__ skip_flag, i64 skip_stride, int* __restrict__ slots) {
  pdl_enter();
  if (blockIdx.y == 0) clear_slot(slots);      // (of one matrix)
  if (skip_flag != nullptr && skip_flag[(i64)blockIdx.y * skip_stride] != 0) return;
  Range g;
  range_scan(g, reinterpret_cast<const float*>(srcs.p[blockIdx.y]), ld, blockIdx.y == 0 ? rows0 : rows1, cols, true,
             (i64)blockIdx.x * 8 + (threadIdx.x >> 5), (i64)gridDim.x * 8);
  block_range(g, part + (i64)blockIdx.y * stride);
}
// M + G into `out` (dense), 4 rows of a warp's 8 x 128 piece at a time, and its range.  VEC as for k_form_b32.
template <bool VEC>
__device__ __forceinline__ void form_sum_range(Range& g, const float* __restrict__ M, i64 ldm, const void* __restrict__ G, i64 ldg, int g_mode,
                                               i64 rows, i64 cols, float* __restrict__ out) {
  const i64 nct = (cols + 127) / 128, pieces = (rows + RANGE_ROWS - 1) / RANGE_ROWS * nct;
  const int lane = threadIdx.x & 31;
  for (i64 w = (i64)blockIdx.x * 8 + (threadIdx.x >> 5); w < pieces; w += (i64)gridDim.x * 8) {
    const i64 tr = row_of(w, nct), c = (w - tr * nct) * 128 + 4 * lane;
    float cm[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int h = 0; h < RANGE_ROWS; h += FORM_BATCH) {
      float4 mv[FORM_BATCH], gv[FORM_BATCH];
#pragma unroll
      for (int u = 0; u < FORM_BATCH; ++u) {
        const i64 i = tr * RANGE_ROWS + h + u;
        mv[u] = gv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (i >= rows || c >= cols) continue;
        const float* mp = M + i * ldm + c;
        mv[u] = VEC ? __ldg(reinterpret_cast<const float4*>(mp)) : make_float4(mp[0], mp[1], mp[2], mp[3]);
        if (g_mode == ADD_F32) {
          const float* gp = reinterpret_cast<const float*>(G) + i * ldg + c;
          gv[u] = VEC ? __ldg(reinterpret_cast<const float4*>(gp)) : make_float4(gp[0], gp[1], gp[2], gp[3]);
        } else if (g_mode == ADD_BF16) {
          const __nv_bfloat16* gp = reinterpret_cast<const __nv_bfloat16*>(G) + i * ldg + c;
          if (VEC) {
            const uint2 t = __ldg(reinterpret_cast<const uint2*>(gp));
            gv[u].x = __uint_as_float(t.x); gv[u].y = __uint_as_float(t.y);
          } else {
            gv[u] = make_float4(__bfloat162float(gp[0]), __bfloat162float(gp[1]), __bfloat162float(gp[2]), __bfloat162float(gp[3]));
          }
        }
      }
#pragma unroll
      for (int u = 0; u < FORM_BATCH; ++u) {
        const i64 i = tr * RANGE_ROWS + h + u;
        float4 v = mv[u], a = gv[u];
        if (VEC && g_mode == ADD_BF16) {      // (still the four bf16 values)
          const uint32_t w0 = __float_as_uint(a.x), w1 = __float_as_uint(a.y);
          a = make_float4(__uint_as_float(w0 << 16), __uint_as_float(w0 & 0xffff0000u), __uint_as_float(w1 << 16), __uint_as_float(w1 & 0xffff0000u));
        }
        if (g_mode != ADD_NONE) { v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w; }
        if (i < rows && c < cols) *reinterpret_cast<float4*>(out + i * cols + c) = v;
        range_row(g, v, cm);
      }
    }
    range_cols(g, cm);
  }
}
// The two launches that prepare a chain (blockIdx.y) of steps on half pairs: M + G in fp32 with the ranges of the sum and of Q
// (Q is a right factor of the caller's making: nothing bounds its entries), then the scaled pairs of both -- or, where the ranges
// say so, a dense fp32 copy of Q for the 3xTF32 product that then forms P, and the sum as a bf16 pair, with which R and the
// error feedback run at the same speed.
// part: gridDim.x partial ranges of the sum (maxima, then minima), then as many of Q.  16-byte accesses to Q where it allows
// them (qvec).
template <bool VEC>
__global__ void __launch_bounds__(256, 3) k_form_sum_amax(const ChainPtrs Ms, i64 ldm, const ChainPtrs Gs, i64 ldg, int g_mode, i64 rows, i64 cols,
                                                       const ChainPtrs Qs, i64 ldq, i64 qrows, i64 qcols, int qvec, float* __restrict__ out,
                                                       float* __restrict__ part, i64 wstride, int* __restrict__ slots, int* __restrict__ flag) {
  pdl_enter();
  clear_slot(slots);
  if (flag != nullptr && blockIdx.x == 0 && threadIdx.x == 0) *flag = 0;      // (the caller's, of one matrix)
  const i64 b = blockIdx.y;
  part += b * wstride;
  Range g, gq;
  form_sum_range<VEC>(g, reinterpret_cast<const float*>(Ms.p[b]), ldm, Gs.p[b], ldg, g_mode, rows, cols, out + b * wstride);
  // (from the last warp down: the first ones have a piece of the sum more)
  range_scan(gq, reinterpret_cast<const float*>(Qs.p[b]), ldq, qrows, qcols, qvec != 0, (i64)gridDim.x * 8 - 1 - ((i64)blockIdx.x * 8 + (threadIdx.x >> 5)),
             (i64)gridDim.x * 8);
  block_range(g, part);
  block_range(gq, part + 2 * gridDim.x);
}
// A step's scalars: the factors that take the scales out of P, R and the error feedback; then R's block maxima.
enum : int { HS_P = 0, HS_R = 1, HS_EF = 2, HS_Q = 3, HS_T = 4, HS_MAX = 16 };      // (HS_Q: 1 / scale of Q; HS_T: Lazy-Dion's left factor)
constexpr int HS_U_BITS = 13;      // U's pair is scaled by 2^13 (entries at most 1)
// eight values as a pair: half values scaled by f (a power of two), or bf16 values as they are
__device__ __forceinline__ void pair_of_8(const float (&x)[8], float f, bool bf16, uint4& hi, uint4& lo) {
  if (!bf16) {
    __half h[8], l[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      h[k] = __float2half_rn(f * x[k]);
      l[k] = __float2half_rn(f * x[k] - __half2float(h[k]));
    }
    hi = *reinterpret_cast<const uint4*>(h); lo = *reinterpret_cast<const uint4*>(l);
  } else {
    uint32_t h[4], l[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      h[k] = pack_bf16x2(x[2 * k], x[2 * k + 1]);
      l[k] = pack_bf16x2(x[2 * k] - __uint_as_float(h[k] << 16), x[2 * k + 1] - __uint_as_float(h[k] & 0xffff0000u));
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]); lo = make_uint4(l[0], l[1], l[2], l[3]);
  }
}
// os (optional: without it the ranges are not looked at): state slots; qd (optional): the dense copy of Q.
__global__ void __launch_bounds__(256) k_split_sum(const float* __restrict__ sum, i64 total_s, const ChainPtrs Qs, i64 ldq, i64 qrows,
                                                   i64 qcols, int qvec, const float* __restrict__ part, int nparts,
                                                   __half* __restrict__ sh, __half* __restrict__ qh, float* __restrict__ qd,
                                                   float* __restrict__ scal, int* __restrict__ os, i64 wstride) {
  pdl_enter();
  const i64 b = blockIdx.y;
  sum += b * wstride; part += b * wstride; scal += b * wstride;
  sh += 2 * b * wstride; qh += 2 * b * wstride;
  const float* __restrict__ Q = reinterpret_cast<const float*>(Qs.p[b]);
  float m0, n0, m1, n1;
  range_of_blocks(part, nparts, m0, n0);
  range_of_blocks(part + 2 * nparts, nparts, m1, n1);
  const bool wide = os != nullptr && range_is_wide(m0, n0, RANGE_UPDATE);
  const bool p32 = os != nullptr && (range_is_wide(m0, n0, RANGE_P) || range_is_wide(m1, n1, RANGE_P));
  const int es = f16_scale_exponent(m0), eq = f16_scale_exponent(m1);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    scal[HS_P] = ldexpf(1.f, -es) * ldexpf(1.f, -eq);
    scal[HS_R] = wide ? 1.f : ldexpf(1.f, -es - HS_U_BITS);
    scal[HS_Q] = ldexpf(1.f, -eq);
    if (os != nullptr) {
      int* o = os + b * OS_SLOT_INTS;
      o[OS_WIDE] = wide ? 1 : 0; o[OS_P32] = p32 ? 1 : 0; o[OS_PHALF] = p32 ? 0 : 1;
    }
  }
  const float fs = ldexpf(1.f, es), fq = ldexpf(1.f, eq);
  const i64 n8 = total_s / 8, qpr = qcols / 8, q8 = qrows * qpr;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < n8 + q8; e += (i64)gridDim.x * blockDim.x) {
    const bool of_q = e >= n8;
    const i64 eo = of_q ? e - n8 : e;
    float4 x, y;
    if (!of_q) {
      x = *reinterpret_cast<const float4*>(sum + eo * 8);
      y = *reinterpret_cast<const float4*>(sum + eo * 8 + 4);
    } else {
      const i64 i = row_of(eo, qpr);
      const float* q = Q + i * ldq + (eo - i * qpr) * 8;
      x = qvec ? *reinterpret_cast<const float4*>(q) : make_float4(q[0], q[1], q[2], q[3]);
      y = qvec ? *reinterpret_cast<const float4*>(q + 4) : make_float4(q[4], q[5], q[6], q[7]);
      if (p32 && qd != nullptr) {
        *reinterpret_cast<float4*>(qd + b * wstride + eo * 8) = x;
        *reinterpret_cast<float4*>(qd + b * wstride + eo * 8 + 4) = y;
        continue;
      }
    }
    const float v[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
    uint4 h, l;
    pair_of_8(v, of_q ? fq : fs, wide && !of_q, h, l);
    __half* hi = (of_q ? qh : sh) + eo * 8;
    *reinterpret_cast<uint4*>(hi) = h;
    *reinterpret_cast<uint4*>(hi + (of_q ? qrows * qcols : total_s)) = l;
  }
}
__global__ void __launch_bounds__(256) k_absmax_partial(const float* __restrict__ src, i64 ld, i64 rows, i64 cols,
                                                        float* __restrict__ part, i64 wstride, const int* __restrict__ skip_flag,
                                                        i64 skip_stride) {
  pdl_enter();
  if (skip_flag != nullptr && skip_flag[(i64)blockIdx.y * skip_stride] != 0) return;
  src += (i64)blockIdx.y * wstride; part += (i64)blockIdx.y * wstride;
  const i64 per_row = cols / 4, total = rows * per_row;
  float m = 0.f;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    const i64 i = row_of(e, per_row), c = (e - i * per_row) * 4;
    const float4 a = *reinterpret_cast<const float4*>(src + i * ld + c);
    m = fmaxf(fmaxf(m, fmaxf(fabsf(a.x), fabsf(a.y))), fmaxf(fabsf(a.z), fabsf(a.w)));
  }
  block_max(m, part);
}
// other_inv < 0: the scalar written is 1 / scale^2 (both operands of the product are this array); else
// other_inv / scale (the other operand carries a fixed scale of its own), times *other_dev when that is given (the
// other operand's own 1 / scale, written by its split; blockIdx.y entries wstride apart like everything else).  own_inv
// (optional): 1 / scale alone.
// os (optional; part holds ranges then: k_range_partial): state slots; the flag u = "wide, or os[in]" (in < 0: wide) goes to
// os[use32] and its opposite to os[usehalf] (both optional, < 0).
__global__ void __launch_bounds__(256) k_split_f16_scaled(const float* __restrict__ src, i64 ld, i64 rows, i64 cols,
                                                          const float* __restrict__ part, int nparts,
                                                          __half* __restrict__ hi, __half* __restrict__ lo,
                                                          float* __restrict__ inv_scale2, i64 wstride,
                                                          const int* __restrict__ skip_flag, i64 skip_stride,
                                                          float other_inv, const float* __restrict__ other_dev, float* __restrict__ own_inv,
                                                          int* __restrict__ os, int in, int use32, int usehalf) {
  pdl_enter();
  if (skip_flag != nullptr && skip_flag[(i64)blockIdx.y * skip_stride] != 0) return;
  src += (i64)blockIdx.y * wstride; part += (i64)blockIdx.y * wstride; inv_scale2 += (i64)blockIdx.y * wstride;
  if (other_dev != nullptr) other_dev += (i64)blockIdx.y * wstride;
  hi += 2 * (i64)blockIdx.y * wstride; lo += 2 * (i64)blockIdx.y * wstride;
  float amax, mn = 0.f;
  if (os != nullptr) {
    range_of_blocks(part, nparts, amax, mn);
  } else {
    __shared__ float red[256];
    float m = 0.f;
    for (int e = threadIdx.x; e < nparts; e += 256) m = fmaxf(m, part[e]);
    red[threadIdx.x] = m;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
      if ((int)threadIdx.x < w) red[threadIdx.x] = fmaxf(red[threadIdx.x], red[threadIdx.x + w]);
      __syncthreads();
    }
    amax = red[0];
  }
  if (os != nullptr && blockIdx.x == 0 && threadIdx.x == 0) {
    os += (i64)blockIdx.y * OS_SLOT_INTS;
    const bool u = range_is_wide(amax, mn, RANGE_P) || (in >= 0 && os[in] != 0);
    if (use32 >= 0) os[use32] = u ? 1 : 0;
    if (usehalf >= 0) os[usehalf] = u ? 0 : 1;
  }
  int ex = 14;                                   // amax = f 2^ex with f in [0.5, 1): scale 2^(14 - ex)
  if (amax > 0.f && amax < 3.0e38f) frexpf(amax, &ex);
  if (ex < -100) ex = -100;
  const float scale = ldexpf(1.f, 14 - ex);
  if (blockIdx.x == 0 && threadIdx.x == 0 && own_inv != nullptr) own_inv[(i64)blockIdx.y * wstride] = ldexpf(1.f, ex - 14);
  if (blockIdx.x == 0 && threadIdx.x == 0)
    *inv_scale2 = (other_inv < 0.f) ? ldexpf(1.f, 2 * (ex - 14))
                                    : other_inv * ldexpf(1.f, ex - 14) * (other_dev != nullptr ? *other_dev : 1.f);
  const i64 per_row = cols / 8, total = rows * per_row;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    const i64 i = row_of(e, per_row), c = (e - i * per_row) * 8;
    const float4 a = *reinterpret_cast<const float4*>(src + i * ld + c);
    const float4 b = *(reinterpret_cast<const float4*>(src + i * ld + c) + 1);
    const float v[8] = {scale * a.x, scale * a.y, scale * a.z, scale * a.w, scale * b.x, scale * b.y, scale * b.z, scale * b.w};
    __half h[8], l[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      h[q] = __float2half_rn(v[q]);
      l[q] = __float2half_rn(v[q] - __half2float(h[q]));
    }
    *reinterpret_cast<uint4*>(hi + i * cols + c) = *reinterpret_cast<const uint4*>(h);
    *reinterpret_cast<uint4*>(lo + i * cols + c) = *reinterpret_cast<const uint4*>(l);
  }
}

// hi = half(scale x), lo = half(scale x - hi) with a scale given by the caller (a power of two; for arrays whose
// entries are bounded, like the unit-norm columns of Q).  Sources from a pointer table (blockIdx.y), outputs
// `ostride` floats apart.
// ldo: leading dimension of the outputs (0: dense).  wide (optional, a state slot apart): flagged matrices get a bf16 pair.
// one (optional, dense): half(scale x) either way.
__global__ void __launch_bounds__(256) k_split_f16_fixed(const ChainPtrs srcs, i64 lds, i64 rows, i64 cols, float scale,
                                                         __half* __restrict__ hi, __half* __restrict__ lo, i64 ostride,
                                                         i64 ldo, const int* __restrict__ skip_flag, i64 skip_stride,
                                                         const int* __restrict__ wide, __half* __restrict__ one) {
  pdl_enter();
  const i64 bm = blockIdx.y;
  if (skip_flag != nullptr && skip_flag[bm * skip_stride] != 0) return;
  if (ldo == 0) ldo = cols;
  const float* __restrict__ src = reinterpret_cast<const float*>(srcs.p[bm]);
  hi += 2 * bm * ostride; lo += 2 * bm * ostride;
  if (one != nullptr) one += 2 * bm * ostride;
  const bool bf16 = wide != nullptr && wide[bm * OS_SLOT_INTS] != 0;
  const i64 per_row = cols / 8, total = rows * per_row;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    const i64 i = row_of(e, per_row), c = (e - i * per_row) * 8;
    const float4 a = *reinterpret_cast<const float4*>(src + i * lds + c);
    const float4 b = *(reinterpret_cast<const float4*>(src + i * lds + c) + 1);
    const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    uint4 h, l;
    pair_of_8(v, scale, bf16, h, l);
    *reinterpret_cast<uint4*>(hi + i * ldo + c) = h;
    *reinterpret_cast<uint4*>(lo + i * ldo + c) = l;
    if (one != nullptr) {
      if (bf16) {
        __half t[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) t[k] = __float2half_rn(scale * v[k]);
        h = *reinterpret_cast<const uint4*>(t);
      }
      *reinterpret_cast<uint4*>(one + i * cols + c) = h;
    }
  }
}

}  // namespace dion
