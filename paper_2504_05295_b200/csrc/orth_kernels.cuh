// Small kernels of the orthonormalization (r x r factor work) and of ColNorm.
#pragma once

#include <cuda_fp16.h>

#include "bf16_kernels.cuh"
#include "chol_flow.cuh"
#include "dion_common.cuh"

namespace dion {

constexpr int NB = CB;  // tile of the factorization

// Round set-up on the r x r Gram matrix G (one block): saves diag(G) to gdiag, writes
// shift = scale * trace(G) (fixed summation order) and resets the round statistics.
// Batched: block b works on the matrix whose scratch starts b * wstride floats further and
// whose state slot is b slots further.
// A trace that is not finite means a NaN or Inf in M, G or Q (every entry of the Gram matrix sums over all
// rows of the panel): the step is cancelled and DION_STATUS_NONFINITE raised.
__global__ void k_round_begin(const float* __restrict__ G, i64 ld, i64 r, float scale,
                              float* __restrict__ gdiag, float* __restrict__ shift,
                              int* __restrict__ os, int adaptive, i64 wstride, int* __restrict__ status) {
  pdl_enter();
  G += (i64)blockIdx.x * wstride; gdiag += (i64)blockIdx.x * wstride; shift += (i64)blockIdx.x * wstride;
  os += (i64)blockIdx.x * OS_SLOT_INTS;
  if (adaptive && os[OS_DONE] != 0) return;
  __shared__ float red[256];
  float s = 0.f;
  for (i64 i = threadIdx.x; i < r; i += blockDim.x) {
    const float v = G[i * ld + i];
    gdiag[i] = v;
    s += v;
  }
  red[threadIdx.x] = s;
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if ((int)threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    *shift = red[0] * scale;
    os[OS_FLOORED] = 0;
    os[OS_MINREL] = 0x7f800000;  // +inf
    if (!(fabsf(red[0]) < __int_as_float(0x7f800000)) && os[OS_FAIL] == 0) {   // (a known failure is not reported twice)
      os[OS_FAIL] = 1;
      atomicOr(status, DION_STATUS_NONFINITE);
    }
  }
}

// CholeskyQR2 of a small panel (rows x r, r <= 64, rows <= TINY_MAX_ROWS, leading dimension r) in ONE launch, one
// CTA of 512 threads per matrix, the panel resident in shared memory: Gram matrix (3xTF32 on the warp-level tensor
// path), Cholesky factor and its inverse (potrf64, on the first eight warps), U1 = P L^-T (3xTF32), then the second round's Gram matrix G2 = U1^T U1, which
// also says exactly how far U1 is from orthonormal: |G2 - I|_F^2 <= tau_f^2 r -> done after one round (the same
// test the probe of the large panels estimates), else the second round runs on G2.  Replaces some seventeen
// launches of a step on such a panel.  Every sum has a fixed order: same bits on every run.
// State as the launch chain leaves it: OS_MAXDEV (the deviation), OS_DONE = 1, OS_ROUNDS and *rounds_total (1 or
// 2); a pivot that is not positive raises OS_FAIL (and DION_STATUS_BREAKDOWN unless `status_fail` is nullptr: a
// fallback follows), the panel is then left to the fallback; a Gram trace that is not finite raises OS_FAIL and
// DION_STATUS_NONFINITE.  Pin may equal Pout.
constexpr int TINY_MAX_ROWS = 512;
constexpr int TINY_THREADS = 512;      // (128 registers a thread: potrf64 keeps an 8 x 8 piece in them)
// Row strides (floats) that keep the fragment loads of the two products off each other's banks: a lane reads
// (row ft, column fg) of the panel for the Gram matrix (stride = 8 mod 32: no conflict) and (row fg, column ft)
// of it and of the inverse (both two-way) for U.
constexpr int TINY_LD = NB + 8;
constexpr int TINY_BLK = CB * CLD;          // floats of a 64 x 64 tile (row stride = 8 mod 32)
inline int tiny_rows_pad(i64 rows) { return (int)((rows + 15) / 16 * 16); }
inline int tiny_cholqr2_smem(i64 rows) {    // panel (rows padded to 16), L, X, red, what potrf64 needs beside them
  return (int)sizeof(float) * (tiny_rows_pad(rows) * TINY_LD + 2 * TINY_BLK + TINY_THREADS) + (int)(sizeof(Potrf64Set) + sizeof(Potrf64Aux));
}

// The two small products of the kernel run on the warp-level tensor-core path (m16n8k8, TF32 operands, fp32
// accumulation) as 3xTF32: x = hi + lo with hi = x truncated to TF32; lo x hi + hi x lo first, hi x hi last.
__device__ __forceinline__ void mma_tf32_16x8x8(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ void split_tf32(float x, uint32_t& hi, uint32_t& lo) {
  hi = __float_as_uint(x) & 0xffffe000u;
  lo = __float_as_uint(x - __uint_as_float(hi));
}
template <int NA, int NB_>
__device__ __forceinline__ void mma_3xtf32(float (&c)[4], const float (&a)[NA], const float (&b)[NB_]) {
  static_assert(NA == 4 && NB_ == 2, "m16n8k8 fragments");
  uint32_t ah[4], al[4], bh[2], bl[2];
#pragma unroll
  for (int x = 0; x < 4; ++x) split_tf32(a[x], ah[x], al[x]);
#pragma unroll
  for (int x = 0; x < 2; ++x) split_tf32(b[x], bh[x], bl[x]);
  mma_tf32_16x8x8(c, al, bh);
  mma_tf32_16x8x8(c, ah, bl);
  mma_tf32_16x8x8(c, ah, bh);
}

__global__ void __launch_bounds__(TINY_THREADS) k_tiny_cholqr2(const float* __restrict__ Pin, float* __restrict__ Pout, int rows, int r,
                                                               int* __restrict__ os, float tau_f, int* __restrict__ rounds_total,
                                                               int* __restrict__ status_fail, int* __restrict__ status_always,
                                                               i64 wstride) {
  Pin += (i64)blockIdx.x * wstride; Pout += (i64)blockIdx.x * wstride;
  os += (i64)blockIdx.x * OS_SLOT_INTS;
  pdl_enter();
  extern __shared__ __align__(16) float tiny_smem[];
  const int rows_pad = (rows + 15) / 16 * 16;
  float* Ps = tiny_smem;                                              // rows_pad x TINY_LD; rows beyond `rows` and columns beyond r are zero
  float* blocks = Ps + rows_pad * TINY_LD;
  ctile_t L = reinterpret_cast<ctile_t>(blocks);
  ctile_t X = reinterpret_cast<ctile_t>(blocks + TINY_BLK);
  float* red = blocks + 2 * TINY_BLK;                                 // TINY_THREADS
  Potrf64Set& set = *reinterpret_cast<Potrf64Set*>(red + TINY_THREADS);
  Potrf64Aux& aux = *reinterpret_cast<Potrf64Aux*>(&set + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int fg = lane >> 2, ft = lane & 3;                            // fragment coordinates of the lane

  if (r % 4 == 0 && (reinterpret_cast<uintptr_t>(Pin) & 15u) == 0) {
    // four 16-byte loads in flight per thread
    const int nv = rows * r / 4;
    const float4* src = reinterpret_cast<const float4*>(Pin);
    for (int base = 0; base < nv; base += TINY_THREADS * 4) {
      float4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int idx = base + u * TINY_THREADS + tid;
        v[u] = (idx < nv) ? __ldg(src + idx) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int idx = base + u * TINY_THREADS + tid;
        if (idx < nv) {
          float* d = Ps + (4 * idx / r) * TINY_LD + (4 * idx % r);
          d[0] = v[u].x; d[1] = v[u].y; d[2] = v[u].z; d[3] = v[u].w;
        }
      }
    }
    if (r < NB)
      for (int e = tid; e < rows * (NB - r); e += TINY_THREADS) Ps[(e / (NB - r)) * TINY_LD + r + e % (NB - r)] = 0.f;
  } else {
#pragma unroll 4
    for (int e = tid; e < rows * NB; e += TINY_THREADS) {
      const int i = e / NB, c = e % NB;
      Ps[i * TINY_LD + c] = (c < r) ? Pin[(i64)i * r + c] : 0.f;
    }
  }
  for (int e = rows * NB + tid; e < rows_pad * NB; e += TINY_THREADS) Ps[(e / NB) * TINY_LD + e % NB] = 0.f;
  __syncthreads();

  // G = P^T P (64 x 64, K = rows_pad): warp w owns the 16 x 8 tiles (w / 4, 2 (w % 4)) and (w / 4, 2 (w % 4) + 1); lane
  // (fg, ft) then holds G[m0 + fg][n0 + 2 ft], [..][n0 + 2 ft + 1], G[m0 + fg + 8][n0 + 2 ft], [..][n0 + 2 ft + 1] of each
  // (n0 = nb0, nb0 + 8).
  const int m0 = (warp >> 2) * 16, nb0 = (warp & 3) * 16;
  float acc[2][4];
  auto gram = [&]() {
#pragma unroll
    for (int t = 0; t < 2; ++t) acc[t][0] = acc[t][1] = acc[t][2] = acc[t][3] = 0.f;
#pragma unroll 4
    for (int k0 = 0; k0 < rows_pad; k0 += 8) {
      const float* r0 = Ps + (k0 + ft) * TINY_LD;
      const float* r1 = Ps + (k0 + ft + 4) * TINY_LD;
      const float a[4] = {r0[m0 + fg], r0[m0 + fg + 8], r1[m0 + fg], r1[m0 + fg + 8]};    // A(m, k) = P[k][m]
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const float b[2] = {r0[nb0 + 8 * t + fg], r1[nb0 + 8 * t + fg]};                  // B(k, n) = P[k][n]
        mma_3xtf32(acc[t], a, b);
      }
    }
  };
  // the Gram matrix from the registers into L: lower triangle, zero above, identity beyond column r; what
  // potrf64 needs beside it
  auto stage_factor_input = [&]() {
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      const int i = m0 + fg + ((x & 2) ? 8 : 0), c = nb0 + 8 * (x >> 2) + 2 * ft + (x & 1);
      if (i == c) red[i] = (i < r) ? acc[x >> 2][x & 3] : 0.f;      // the diagonal (also for the trace)
    }
    __syncthreads();
    if (warp == 0) potrf64_setup(set, red[lane], red[lane + 32], 0.f, lane);
    __syncthreads();
    const float s2 = set.s2;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      const int i = m0 + fg + ((x & 2) ? 8 : 0), c = nb0 + 8 * (x >> 2) + 2 * ft + (x & 1);
      float v = (i < r && c <= i) ? acc[x >> 2][x & 3] * s2 : 0.f;
      if (i == c && i >= r) v = 1.f;
      L[i][c] = v;
    }
  };
  // U = P X^T in place (X lower triangular, its zeros above the diagonal stored): work item = 16 rows x 32
  // columns, K = 64; the items of a sweep are all computed before any entry of the panel is overwritten.
  auto apply_inverse = [&]() {
    const int items = (rows_pad / 16) * 2;
    for (int it0 = 0; it0 < items; it0 += TINY_THREADS / 32) {
      const int it = it0 + warp;
      const int i0 = (it >> 1) * 16, c0 = (it & 1) * 32;
      float y[4][4];
#pragma unroll
      for (int nt = 0; nt < 4; ++nt) y[nt][0] = y[nt][1] = y[nt][2] = y[nt][3] = 0.f;
      if (it < items) {
#pragma unroll 2
        for (int k0 = 0; k0 < NB; k0 += 8) {
          const float* r0 = Ps + (i0 + fg) * TINY_LD + k0;
          const float* r1 = Ps + (i0 + fg + 8) * TINY_LD + k0;
          const float a[4] = {r0[ft], r1[ft], r0[ft + 4], r1[ft + 4]};                    // A(m, k) = P[i0 + m][k]
#pragma unroll
          for (int nt = 0; nt < 4; ++nt) {
            const float* xr = &X[c0 + 8 * nt + fg][k0];
            const float b[2] = {xr[ft], xr[ft + 4]};                                      // B(k, n) = X[n][k]
            mma_3xtf32(y[nt], a, b);
          }
        }
      }
      __syncthreads();
      if (it < items) {
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) {
          const int c = c0 + 8 * nt + 2 * ft;
          float* w0 = Ps + (i0 + fg) * TINY_LD + c;
          float* w1 = Ps + (i0 + fg + 8) * TINY_LD + c;
          w0[0] = y[nt][0]; w0[1] = y[nt][1]; w1[0] = y[nt][2]; w1[1] = y[nt][3];
        }
      }
    }
    __syncthreads();
  };

  gram();
  stage_factor_input();
  __syncthreads();
  if (warp == 8) {      // (a warp that has no part in the factorization: the trace from the staged diagonal, fixed order)
    float tr = red[lane] + red[lane + 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tr += __shfl_xor_sync(0xffffffffu, tr, o);
    if (lane == 0 && !(fabsf(tr) < __int_as_float(0x7f800000)) && os[OS_FAIL] == 0) {
      os[OS_FAIL] = 1;
      atomicOr(status_always, DION_STATUS_NONFINITE);
    }
  }
  if (tid < 256) potrf64(L, X, set, aux, 0.f, os, status_fail, tid);   // (ends with its own barrier)
  __syncthreads();
  const bool failed1 = reinterpret_cast<volatile int*>(os)[OS_FAIL] != 0;   // (written by this CTA's thread 0 before that barrier, or before this launch)
  apply_inverse();

  // the second round's Gram matrix, and with it the first round's distance from orthonormal
  gram();
  float e = 0.f;
#pragma unroll
  for (int x = 0; x < 8; ++x) {
    const int i = m0 + fg + ((x & 2) ? 8 : 0), c = nb0 + 8 * (x >> 2) + 2 * ft + (x & 1);
    if (i < r && c < r) { const float d = acc[x >> 2][x & 3] - ((i == c) ? 1.f : 0.f); e = fmaf(d, d, e); }
  }
  red[tid] = e;
  __syncthreads();
  for (int w = TINY_THREADS / 2; w > 0; w >>= 1) {
    if (tid < w) red[tid] += red[tid + w];
    __syncthreads();
  }
  const float est = red[0];
  const bool done = !failed1 && (est <= tau_f * tau_f * (float)r);      // false for NaN
  if (!done && !failed1) {
    __syncthreads();                 // everyone has read red[0]
    stage_factor_input();
    __syncthreads();
    if (tid < 256) potrf64(L, X, set, aux, 0.f, os, status_fail, tid);
    __syncthreads();
    apply_inverse();
  }
  if (tid == 0) {
    os[OS_MAXDEV] = __float_as_int(est);
    os[OS_DONE] = 1;
    os[OS_ROUNDS] = done ? 1 : 2;
    atomicAdd(rounds_total, done ? 1 : 2);
  }
#pragma unroll 4
  for (int e2 = tid; e2 < rows * r; e2 += TINY_THREADS) {
    const int i = e2 / r, c = e2 % r;
    Pout[(i64)i * r + c] = Ps[i * TINY_LD + c];
  }
}

// The finishing round of a panel that is orthonormal already but for a small defect E (its Gram matrix is I + E): the inverse
// of its triangular factor, transposed, is a short series
//   X = L^-T = I - Phi^T + Psi^T + O(E^3),  Phi = strictly lower part of E + half its diagonal,
//   Psi = strictly lower part of S = Phi E, its diagonal (S_ii + Phi_ii^2) / 2
// (from L L^T = I + E order by order).  Where |E|_F <= max_def and the last round was good (OS_GOOD == 1) this kernel
// leaves scale x E and scale x Phi as IEEE half arrays for the product S (the second-order term needs few bits) and
// sets OS_GOOD to 2: the factorization's launch then leaves the matrix alone and k_split_f16_tri puts X together.
// (At r = 2048 that launch takes 390 us, this and the product 35.)  Else OS_NOTNEAR is set: the product is skipped.
// A panel whose range is too wide for its pair (OS_PANEL_WIDE) is solved by substitution instead.
// Gram matrix: `part` (nsplit partial sums, times *alpha_dev) or G, lower triangle, r a multiple of 8.
// grid = (blocks, matrices), 256 threads, a 32 x 32 tile at a time; sums: one float per block; OS_BARRIER as in k_probe_decide.
struct NearSrc {
  const float* G; const float* part; int nsplit; const float* alpha_dev;
};
__device__ __forceinline__ float4 near_load(const NearSrc& g, i64 wo, i64 r, i64 i, i64 j) {      // four entries of E + I
  if (g.nsplit <= 1) return *reinterpret_cast<const float4*>(g.G + wo + i * r + j);
  const float* p = g.part + wo + i * r + j;
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int q = 0; q < g.nsplit; ++q, p += r * r) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
  }
  const float a = (g.alpha_dev != nullptr) ? g.alpha_dev[wo] : 1.f;
  return make_float4(s.x * a, s.y * a, s.z * a, s.w * a);
}
constexpr float NEAR_SCALE = 4096.f;
__global__ void __launch_bounds__(256) k_near_identity(const NearSrc g, i64 r, __half* __restrict__ Eh, __half* __restrict__ Ph,
                                                       float* __restrict__ xmax, float* __restrict__ sums, int* __restrict__ os, float max_def,
                                                       i64 wstride) {
  pdl_enter();
  os += (i64)blockIdx.y * OS_SLOT_INTS;
  if (os[OS_DONE] != 0 || os[OS_GOOD] != 1 || os[OS_PANEL_WIDE] != 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) os[OS_NOTNEAR] = 1;
    return;
  }
  const i64 wo = (i64)blockIdx.y * wstride;
  Eh += 2 * wo; Ph += 2 * wo; xmax += wo; sums += wo;
  __shared__ float T[32][33];
  __shared__ float red[8];
  __shared__ int s_last;
  const int row = threadIdx.x >> 3, c4 = (threadIdx.x & 7) * 4, lane = threadIdx.x & 31;
  const int n = (int)((r + 31) / 32);
  float e2 = 0.f;
  auto put = [&](__half* dst, const float (&v)[4]) {
    __half2 a = __floats2half2_rn(NEAR_SCALE * v[0], NEAR_SCALE * v[1]), b = __floats2half2_rn(NEAR_SCALE * v[2], NEAR_SCALE * v[3]);
    uint2 u;
    u.x = *reinterpret_cast<uint32_t*>(&a); u.y = *reinterpret_cast<uint32_t*>(&b);
    *reinterpret_cast<uint2*>(dst) = u;
  };
  for (i64 q = blockIdx.x; q < (i64)n * n; q += gridDim.x) {
    const int ti = (int)(q / n), tj = (int)(q % n);
    if (tj > ti) continue;
    const i64 i = (i64)ti * 32 + row, j = (i64)tj * 32 + c4;
    float e[4] = {0.f, 0.f, 0.f, 0.f}, ph[4];
    if (i < r && j < r) {
      const float4 v = near_load(g, wo, r, i, j);
      e[0] = v.x; e[1] = v.y; e[2] = v.z; e[3] = v.w;
    }
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      if (j + x > i) e[x] = 0.f;
      if (j + x == i) e[x] -= 1.f;
      if (i >= r || j >= r) e[x] = 0.f;
      e2 = fmaf((i == j + x) ? e[x] : 2.f * e[x], e[x], e2);
      ph[x] = (i == j + x) ? 0.5f * e[x] : e[x];
      T[row][c4 + x] = e[x];
    }
    __syncthreads();
    if (i < r && j < r) {
      put(Ph + i * r + j, ph);
      if (ti == tj) {
        float f[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) f[x] = (j + x > i) ? T[c4 + x][row] : e[x];
        put(Eh + i * r + j, f);
      } else {
        put(Eh + i * r + j, e);
      }
    }
    if (ti != tj) {      // the mirror tile (tj, ti)
      const i64 mi = (i64)tj * 32 + row, mj = (i64)ti * 32 + c4;
      if (mi < r && mj < r) {
        float f[4];
        const float z[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int x = 0; x < 4; ++x) f[x] = T[c4 + x][row];
        put(Eh + mi * r + mj, f);
        put(Ph + mi * r + mj, z);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e2 += __shfl_xor_sync(0xffffffffu, e2, o);
  if (lane == 0) red[threadIdx.x >> 5] = e2;
  __syncthreads();
  if (threadIdx.x == 0) {
    sums[blockIdx.x] = ((red[0] + red[1]) + (red[2] + red[3])) + ((red[4] + red[5]) + (red[6] + red[7]));
    __threadfence();
    s_last = (atomicAdd(&os[OS_BARRIER], 1) == (int)gridDim.x - 1) ? 1 : 0;
  }
  __syncthreads();
  if (s_last == 0 || threadIdx.x >= 32) return;
  __threadfence();
  float t = 0.f;
  for (int c = lane; c < (int)gridDim.x; c += 32) t += __ldcg(sums + c);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) {
    os[OS_BARRIER] = 0;
    os[OS_MAXDEV] = __float_as_int(t);
    const bool near = t <= max_def * max_def;      // (false for NaN)
    os[OS_NOTNEAR] = near ? 0 : 1;
    if (near) {
      *xmax = 1.f + max_def;
      os[OS_GOOD] = 2;
    }
  }
}

// The scaled half pair of X = L^-T (n x n, upper triangular, n a multiple of 8) as far down each column as a product of
// 256-column tiles reads: from src, or, with S given, put together from the Gram matrix and S (k_near_identity).
// Scale as in k_split_f16_scaled from *amax, the largest magnitude.  *inv_out = 1 / scale, times the root of *other_sq (a power
// of four: the square of the other operand's 1 / scale).  grid = (blocks, matrices), 256 threads, 32 x 32 tiles.
// os (optional): state slots; OS_USE32 and OS_USEHALF say which product takes the panel to U: the one on the pairs, or the
// 3xTF32 one where the panel or the columns of X (its diagonal: no column's largest entry is smaller) spread over more than the
// pairs hold (see k_form_sum_amax); neither when the round is skipped.
__global__ void __launch_bounds__(256) k_split_f16_tri(const float* __restrict__ src, i64 n, const float* __restrict__ amax,
                                                       const float* __restrict__ other_sq, __half* __restrict__ hi, __half* __restrict__ lo,
                                                       float* __restrict__ inv_out, i64 wstride, const int* __restrict__ skip_flag,
                                                       const NearSrc g, const float* __restrict__ S, int* __restrict__ os) {
  pdl_enter();
  if (os != nullptr) os += (i64)blockIdx.y * OS_SLOT_INTS;
  if (skip_flag != nullptr && skip_flag[(i64)blockIdx.y * OS_SLOT_INTS] != 0) {
    if (os != nullptr && blockIdx.x == 0 && threadIdx.x == 0) os[OS_USE32] = os[OS_USEHALF] = 1;
    return;
  }
  const bool near = S != nullptr;
  const i64 wo = (i64)blockIdx.y * wstride;
  src += wo; hi += 2 * wo; lo += 2 * wo;
  if (S != nullptr) S += wo;
  const float m = amax[wo];
  if (os != nullptr && blockIdx.x == 0) {
    bool u = os[OS_PANEL_WIDE] != 0;
    for (i64 i = threadIdx.x; i < n; i += 256) u = u || fabsf(src[i * n + i]) < m * RANGE_P;
    u = __syncthreads_or(u) != 0;
    if (threadIdx.x == 0) { os[OS_USE32] = u ? 1 : 0; os[OS_USEHALF] = u ? 0 : 1; }
  }
  int ex = 14;                                   // amax = f 2^ex with f in [0.5, 1): scale 2^(14 - ex)
  if (m > 0.f && m < 3.0e38f) frexpf(m, &ex);
  if (ex < -100) ex = -100;
  const float scale = ldexpf(1.f, 14 - ex);
  if (blockIdx.x == 0 && threadIdx.x == 0) inv_out[wo] = ldexpf(1.f, ex - 14) * sqrtf(other_sq[wo]);
  __shared__ float T[32][33];
  const int row = threadIdx.x >> 3, c4 = (threadIdx.x & 7) * 4;
  const int nt = (int)((n + 31) / 32);
  for (i64 q = blockIdx.x; q < (i64)nt * nt; q += gridDim.x) {
    const int tk = (int)(q / nt), tc = (int)(q % nt);      // tile of X: rows tk, columns tc
    if (tk > tc / 8 * 8 + 7) continue;
    const i64 k = (i64)tk * 32 + row, c = (i64)tc * 32 + c4;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    if (near) {
      const i64 i = (i64)tc * 32 + row, j = (i64)tk * 32 + c4;      // the lower tile (tc, tk)
      float4 e = make_float4(0.f, 0.f, 0.f, 0.f), s = e;
      if (tk <= tc && i < n && j < n) {
        e = near_load(g, wo, n, i, j);
        s = *reinterpret_cast<const float4*>(S + i * n + j);
      }
      const float ev[4] = {e.x, e.y, e.z, e.w}, sv[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const float d = ev[x] - 1.f;
        T[row][c4 + x] = (j + x < i) ? sv[x] - ev[x] : (j + x == i) ? 1.f - 0.5f * d + 0.5f * (sv[x] + 0.25f * d * d) : 0.f;
      }
      __syncthreads();
#pragma unroll
      for (int x = 0; x < 4; ++x) v[x] = T[c4 + x][row];
      __syncthreads();
    } else if (k < n && c < n) {
      const float4 a = *reinterpret_cast<const float4*>(src + k * n + c);
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    }
    if (k >= n || c >= n) continue;
    __half h[4], l[4];
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const float y = scale * v[x];
      h[x] = __float2half_rn(y);
      l[x] = __float2half_rn(y - __half2float(h[x]));
    }
    *reinterpret_cast<uint2*>(hi + k * n + c) = *reinterpret_cast<const uint2*>(h);
    *reinterpret_cast<uint2*>(lo + k * n + c) = *reinterpret_cast<const uint2*>(l);
  }
}

// End of an adaptive round for the matrices that took the series (one thread per matrix).
__global__ void k_near_end(int* __restrict__ os, int* __restrict__ rounds_total) {
  pdl_enter();
  os += (i64)blockIdx.x * OS_SLOT_INTS;
  if (os[OS_DONE] != 0 || os[OS_GOOD] != 2) return;
  os[OS_ROUNDS] += 1;
  atomicAdd(rounds_total, 1);
  os[OS_DONE] = 1;
}

// End of an adaptive round whose panel was solved by products behind the factorization (one thread per matrix).
__global__ void k_round_end(int* __restrict__ os, float good_rel, float done_rel, int* __restrict__ rounds_total) {
  pdl_enter();
  os += (i64)blockIdx.x * OS_SLOT_INTS;
  if (os[OS_DONE] != 0) return;
  round_evaluate(os, good_rel, done_rel, rounds_total);
}

// ---------------------------------------------------------------------------
// CholeskyQR2: is the first round's result U1 orthonormal enough to skip the second?  Measured without forming
// U1^T U1 (one third of the orthonormalization's tensor work): with NPROBE fixed sign vectors z_p (entries +-1
// from a hash of the index), E = U1^T U1 - I and w_p = U1^T (U1 z_p),  sum_p |w_p - z_p|^2 / NPROBE  is an
// unbiased estimate of |E|_F^2 (Hutchinson's estimator; relative spread sqrt(2 / NPROBE) per probe set at
// worst, far less for a matrix whose weight is spread over many entries).  Two passes over the panel.
// ---------------------------------------------------------------------------
constexpr int NPROBE = 8;

__device__ __forceinline__ float probe_sign(i64 j, int p) {
  uint32_t h = (uint32_t)j * 2654435761u + (uint32_t)(p + 1) * 0x9E3779B9u;
  h ^= h >> 15; h *= 2246822519u; h ^= h >> 13; h *= 3266489917u; h ^= h >> 16;
  return (h & 1u) ? 1.f : -1.f;
}

// Y[i][p] = sum_j U[i][j] z_p[j]: one warp per row (lanes stride over the columns).  grid = (blocks, matrices).
__global__ void __launch_bounds__(256) k_probe_y(const float* __restrict__ U, i64 ld, i64 rows, i64 r,
                                                 float* __restrict__ Y, i64 wstride, const int* __restrict__ keep) {
  pdl_enter();
  if (keep != nullptr && keep[(i64)blockIdx.y * OS_SLOT_INTS] != 0) return;   // this panel's decision stands
  U += (i64)blockIdx.y * wstride; Y += (i64)blockIdx.y * wstride;
  const int lane = threadIdx.x & 31;
  const i64 warp = (i64)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const i64 nwarps = (i64)gridDim.x * (blockDim.x >> 5);
  for (i64 i = warp; i < rows; i += nwarps) {
    float acc[NPROBE];
#pragma unroll
    for (int p = 0; p < NPROBE; ++p) acc[p] = 0.f;
    const float* urow = U + i * ld;
    for (i64 j = lane; j < r; j += 32) {
      const float u = urow[j];
#pragma unroll
      for (int p = 0; p < NPROBE; ++p) acc[p] = fmaf(u, probe_sign(j, p), acc[p]);
    }
#pragma unroll
    for (int p = 0; p < NPROBE; ++p) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[p] += __shfl_xor_sync(0xffffffffu, acc[p], o);
    }
    if (lane == 0) {
#pragma unroll
      for (int p = 0; p < NPROBE; ++p) Y[i * NPROBE + p] = acc[p];
    }
  }
}

// The same for wider panels (r a multiple of 4 above PF_MAX_R; 16-byte aligned rows): the +-1 entries of the probe vectors are hashed once per
// CTA and column block into a shared-memory table of floats instead of once per matrix element (the hash made the
// plain kernel ALU bound at a seventh of HBM speed), and a warp takes four rows at a time so that one read of a
// column's eight signs serves four elements.  Lane l owns columns 128 t + 4 l .. + 3 of a block of PY_COLS
// columns; wider panels add their later column blocks into Y (the same warp owns a row throughout).
constexpr int PY_COLS = 2048;
constexpr int PY_SMEM = PY_COLS * NPROBE * 4;
__global__ void __launch_bounds__(256) k_probe_y4(const float* __restrict__ U, i64 ld, i64 rows, i64 r,
                                                  float* __restrict__ Y, i64 wstride, const int* __restrict__ keep) {
  extern __shared__ __align__(16) float py_sign[];      // the signs of the block's columns (layout below)
  pdl_enter();
  if (keep != nullptr && keep[(i64)blockIdx.y * OS_SLOT_INTS] != 0) return;   // this panel's decision stands
  U += (i64)blockIdx.y * wstride; Y += (i64)blockIdx.y * wstride;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const i64 group0 = (i64)blockIdx.x * 8 + warp, groups = (i64)gridDim.x * 8;
  for (i64 c0 = 0; c0 < r; c0 += PY_COLS) {
    const int nc = (int)min((i64)PY_COLS, r - c0);
    __syncthreads();
    // table layout: the four signs (probes 4 h .. 4 h + 3) of column 128 t + 4 l + cc sit in the 16-byte unit
    // ((4 t + cc) 2 + h) 32 + l, so that the 32 lanes of a warp read 32 consecutive units (column-major by 8 floats
    // put a quarter warp's reads on the same banks: eight-way conflicts on every read)
    for (int e = threadIdx.x; e < nc * NPROBE; e += 256) {
      const int col = e / NPROBE, pr = e % NPROBE;
      py_sign[((((col >> 7) * 4 + (col & 3)) * 2 + (pr >> 2)) * 32 + ((col & 127) >> 2)) * 4 + (pr & 3)] = probe_sign(c0 + col, pr);
    }
    __syncthreads();
    for (i64 g = group0; g * 4 < rows; g += groups) {
      const i64 i0 = g * 4;
      float acc[4][NPROBE];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int p = 0; p < NPROBE; ++p) acc[q][p] = 0.f;
      for (int j = 4 * lane; j < nc; j += 128) {
        float4 u[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          u[q] = (i0 + q < rows) ? *reinterpret_cast<const float4*>(U + (i0 + q) * ld + c0 + j) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int cc = 0; cc < 4; ++cc) {
          const float4* su = reinterpret_cast<const float4*>(py_sign) + (((j >> 7) * 4 + cc) * 2) * 32 + lane;
          const float4 s0 = su[0];
          const float4 s1 = su[32];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const float v = (cc == 0) ? u[q].x : (cc == 1) ? u[q].y : (cc == 2) ? u[q].z : u[q].w;
            acc[q][0] = fmaf(v, s0.x, acc[q][0]); acc[q][1] = fmaf(v, s0.y, acc[q][1]);
            acc[q][2] = fmaf(v, s0.z, acc[q][2]); acc[q][3] = fmaf(v, s0.w, acc[q][3]);
            acc[q][4] = fmaf(v, s1.x, acc[q][4]); acc[q][5] = fmaf(v, s1.y, acc[q][5]);
            acc[q][6] = fmaf(v, s1.z, acc[q][6]); acc[q][7] = fmaf(v, s1.w, acc[q][7]);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int p = 0; p < NPROBE; ++p) {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) acc[q][p] += __shfl_xor_sync(0xffffffffu, acc[q][p], o);
        }
      if (lane < 4 && i0 + lane < rows) {
        float* y = Y + (i0 + lane) * NPROBE;
#pragma unroll
        for (int p = 0; p < NPROBE; ++p) {
          const float v = (lane == 0) ? acc[0][p] : (lane == 1) ? acc[1][p] : (lane == 2) ? acc[2][p] : acc[3][p];
          y[p] = (c0 == 0) ? v : y[p] + v;
        }
      }
    }
  }
}

// part[chunk][j][p] = sum over the chunk's rows of U[i][j] Y[i][p].  grid = (ceil(r/128), chunks, matrices).
__global__ void __launch_bounds__(128) k_probe_w(const float* __restrict__ U, i64 ld, i64 rows, i64 r,
                                                 i64 rows_per_chunk, const float* __restrict__ Y,
                                                 float* __restrict__ part, i64 wstride, const int* __restrict__ keep) {
  pdl_enter();
  if (keep != nullptr && keep[(i64)blockIdx.z * OS_SLOT_INTS] != 0) return;
  U += (i64)blockIdx.z * wstride; Y += (i64)blockIdx.z * wstride; part += (i64)blockIdx.z * wstride;
  const i64 j = (i64)blockIdx.x * 128 + threadIdx.x;
  if (j >= r) return;
  const i64 i0 = (i64)blockIdx.y * rows_per_chunk;
  const i64 i1 = min(rows, i0 + rows_per_chunk);
  float acc[NPROBE];
#pragma unroll
  for (int p = 0; p < NPROBE; ++p) acc[p] = 0.f;
#pragma unroll 8      // (eight rows' loads in flight per thread; the sums keep their order)
  for (i64 i = i0; i < i1; ++i) {
    const float u = U[i * ld + j];
    const float4 y0 = *reinterpret_cast<const float4*>(Y + i * NPROBE);
    const float4 y1 = *reinterpret_cast<const float4*>(Y + i * NPROBE + 4);
    acc[0] = fmaf(u, y0.x, acc[0]); acc[1] = fmaf(u, y0.y, acc[1]); acc[2] = fmaf(u, y0.z, acc[2]); acc[3] = fmaf(u, y0.w, acc[3]);
    acc[4] = fmaf(u, y1.x, acc[4]); acc[5] = fmaf(u, y1.y, acc[5]); acc[6] = fmaf(u, y1.z, acc[6]); acc[7] = fmaf(u, y1.w, acc[7]);
  }
  float* out = part + ((i64)blockIdx.y * r + j) * NPROBE;
#pragma unroll
  for (int p = 0; p < NPROBE; ++p) out[p] = acc[p];
}

// The same for wide panels, r a multiple of 4: a thread takes four neighbouring columns (one 16-byte load per row, eight rows'
// loads in flight); every column's sum runs over the chunk's rows in the same order as above.
// grid = (ceil(r/512), chunks, matrices).
__global__ void __launch_bounds__(128) k_probe_w4(const float* __restrict__ U, i64 ld, i64 rows, i64 r,
                                                  i64 rows_per_chunk, const float* __restrict__ Y,
                                                  float* __restrict__ part, i64 wstride, const int* __restrict__ keep) {
  pdl_enter();
  if (keep != nullptr && keep[(i64)blockIdx.z * OS_SLOT_INTS] != 0) return;
  U += (i64)blockIdx.z * wstride; Y += (i64)blockIdx.z * wstride; part += (i64)blockIdx.z * wstride;
  const i64 j = ((i64)blockIdx.x * 128 + threadIdx.x) * 4;
  if (j >= r) return;
  const i64 i0 = (i64)blockIdx.y * rows_per_chunk;
  const i64 i1 = min(rows, i0 + rows_per_chunk);
  float acc[4][NPROBE];
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int p = 0; p < NPROBE; ++p) acc[c][p] = 0.f;
#pragma unroll 8
  for (i64 i = i0; i < i1; ++i) {
    const float4 u4 = *reinterpret_cast<const float4*>(U + i * ld + j);
    const float4 y0 = *reinterpret_cast<const float4*>(Y + i * NPROBE);
    const float4 y1 = *reinterpret_cast<const float4*>(Y + i * NPROBE + 4);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float u = (c == 0) ? u4.x : (c == 1) ? u4.y : (c == 2) ? u4.z : u4.w;
      acc[c][0] = fmaf(u, y0.x, acc[c][0]); acc[c][1] = fmaf(u, y0.y, acc[c][1]);
      acc[c][2] = fmaf(u, y0.z, acc[c][2]); acc[c][3] = fmaf(u, y0.w, acc[c][3]);
      acc[c][4] = fmaf(u, y1.x, acc[c][4]); acc[c][5] = fmaf(u, y1.y, acc[c][5]);
      acc[c][6] = fmaf(u, y1.z, acc[c][6]); acc[c][7] = fmaf(u, y1.w, acc[c][7]);
    }
  }
  float4* out = reinterpret_cast<float4*>(part + ((i64)blockIdx.y * r + j) * NPROBE);
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    out[2 * c] = make_float4(acc[c][0], acc[c][1], acc[c][2], acc[c][3]);
    out[2 * c + 1] = make_float4(acc[c][4], acc[c][5], acc[c][6], acc[c][7]);
  }
}

// Both passes in one launch for r up to PF_MAX_R: a block takes 32 rows at a time (they stay in L1 between the
// passes), its warps four rows each for Y = U z, then (1 << ct_log) threads by four columns and the rest by row groups for
// U^T Y.  Two launches read the panel twice from L2 and met in memory: 2048 x 128 14.5 us, 4096 x 1024 23 us (now 5 and 15 us).
// VEC: r a multiple of 4 (rows on 16-byte boundaries); other r read entry by entry (1001 x 83: the step 119.8 -> 113.8 us).
// grid = (chunks, matrices); part[chunk][j][p] as in k_probe_w.
constexpr i64 PF_MAX_R = 1024;      // 256 threads by four columns
constexpr int PF_RED = 256 * 4 * NPROBE;      // floats: row groups x columns x probes
constexpr int PF_SMEM_MAX = ((int)PF_MAX_R * NPROBE + PF_RED + 32 * NPROBE) * 4;
template <bool VEC>
__global__ void __launch_bounds__(256) k_probe_fused(const float* __restrict__ U, i64 ld, i64 rows, i64 r, i64 rows_per_chunk,
                                                     float* __restrict__ part, i64 wstride, const int* __restrict__ keep, int ct_log) {
  extern __shared__ __align__(16) float pf_smem[];
  pdl_enter();
  if (keep != nullptr && keep[(i64)blockIdx.y * OS_SLOT_INTS] != 0) return;   // this panel's decision stands
  U += (i64)blockIdx.y * wstride; part += (i64)blockIdx.y * wstride;
  float* ys = pf_smem;                             // [32][NPROBE]
  float* red = ys + 32 * NPROBE;                   // [row group][column][probe]
  float* sign = red + PF_RED;                      // (layout of k_probe_y4)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nr = (int)r;
  for (int e = threadIdx.x; e < (nr + 3) / 4 * 4 * NPROBE; e += 256) {
    const int col = e / NPROBE, pr = e % NPROBE;
    sign[((((col >> 7) * 4 + (col & 3)) * 2 + (pr >> 2)) * 32 + ((col & 127) >> 2)) * 4 + (pr & 3)] = probe_sign(col, pr);
  }
  __syncthreads();
  auto row4 = [&](const float* p, int j) -> float4 {      // columns j .. j + 3 of a row
    if (VEC) return *reinterpret_cast<const float4*>(p);
    return make_float4(p[0], j + 1 < nr ? p[1] : 0.f, j + 2 < nr ? p[2] : 0.f, j + 3 < nr ? p[3] : 0.f);
  };
  const int groups = 256 >> ct_log, per = 32 / groups;      // row groups, rows of each (groups <= 32)
  const int j0 = 4 * ((int)threadIdx.x & ((1 << ct_log) - 1)), grp = (int)threadIdx.x >> ct_log;
  float w[4][NPROBE];
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int p = 0; p < NPROBE; ++p) w[c][p] = 0.f;
  const i64 b0 = (i64)blockIdx.x * rows_per_chunk, b1 = min(rows, b0 + rows_per_chunk);
  for (i64 ib = b0; ib < b1; ib += 32) {
    float acc[4][NPROBE];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int p = 0; p < NPROBE; ++p) acc[q][p] = 0.f;
    const i64 i0 = ib + 4 * warp;
    for (int j = 4 * lane; j < nr; j += 128) {
      float4 v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
        v[q] = (i0 + q < b1) ? row4(U + (i0 + q) * ld + j, j) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        const float4* su = reinterpret_cast<const float4*>(sign) + (((j >> 7) * 4 + cc) * 2) * 32 + lane;
        const float4 s0 = su[0], s1 = su[32];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float x = (cc == 0) ? v[q].x : (cc == 1) ? v[q].y : (cc == 2) ? v[q].z : v[q].w;
          acc[q][0] = fmaf(x, s0.x, acc[q][0]); acc[q][1] = fmaf(x, s0.y, acc[q][1]);
          acc[q][2] = fmaf(x, s0.z, acc[q][2]); acc[q][3] = fmaf(x, s0.w, acc[q][3]);
          acc[q][4] = fmaf(x, s1.x, acc[q][4]); acc[q][5] = fmaf(x, s1.y, acc[q][5]);
          acc[q][6] = fmaf(x, s1.z, acc[q][6]); acc[q][7] = fmaf(x, s1.w, acc[q][7]);
        }
      }
    }
    // the 32 sums of the warp (4 rows x 8 probes): lane l ends up with sum l (each step halves what a lane still holds)
    float v32[32];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int p = 0; p < NPROBE; ++p) v32[q * NPROBE + p] = acc[q][p];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int k = 0; k < o; ++k) {
        const float send = up ? v32[k] : v32[k + o], mine = up ? v32[k + o] : v32[k];
        v32[k] = mine + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    ys[warp * 32 + lane] = v32[0];      // (row 4 warp + lane / 8, probe lane % 8)
    __syncthreads();
    if (j0 < nr) {
#pragma unroll 4
      for (int q = 0; q < per; ++q) {
        const int i = grp * per + q;
        if (ib + i >= b1) break;
        const float4 u4 = row4(U + (ib + i) * ld + j0, j0);
        const float4 y0 = *reinterpret_cast<const float4*>(ys + i * NPROBE), y1 = *reinterpret_cast<const float4*>(ys + i * NPROBE + 4);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float x = (c == 0) ? u4.x : (c == 1) ? u4.y : (c == 2) ? u4.z : u4.w;
          w[c][0] = fmaf(x, y0.x, w[c][0]); w[c][1] = fmaf(x, y0.y, w[c][1]); w[c][2] = fmaf(x, y0.z, w[c][2]); w[c][3] = fmaf(x, y0.w, w[c][3]);
          w[c][4] = fmaf(x, y1.x, w[c][4]); w[c][5] = fmaf(x, y1.y, w[c][5]); w[c][6] = fmaf(x, y1.z, w[c][6]); w[c][7] = fmaf(x, y1.w, w[c][7]);
        }
      }
    }
    __syncthreads();
  }
  if (j0 < nr) {
    float4* out = reinterpret_cast<float4*>(groups > 1 ? red + ((grp << ct_log) * 4 + j0) * NPROBE : part + ((i64)blockIdx.x * r + j0) * NPROBE);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (!VEC && groups == 1 && j0 + c >= nr) break;
      out[2 * c] = make_float4(w[c][0], w[c][1], w[c][2], w[c][3]);
      out[2 * c + 1] = make_float4(w[c][4], w[c][5], w[c][6], w[c][7]);
    }
  }
  if (groups == 1) return;
  __syncthreads();
  for (int e = threadIdx.x; e < nr * NPROBE; e += 256) {
    float s = 0.f;
    for (int g = 0; g < groups; ++g) s += red[((g << ct_log) * 4) * NPROBE + e];
    part[(i64)blockIdx.x * r * NPROBE + e] = s;
  }
}

// est = sum_p |w_p - z_p|^2 / NPROBE (fixed summation order) into os[OS_MAXDEV] (float bits); est <= tau_f^2 * r  ->  the
// panel is done (OS_DONE = 1: the rest of the second round is skipped).
// Counts the rounds of the step that did work (1 or 2; with a recomputed panel 2 or 3).
// phase PROBE_FAST (the round ran on a panel from the fast product): done -> OS_DONE = 1, else 0 (a failed pivot
// too: the panel is recomputed before the fallback sees it); nothing is counted.  PROBE_AFTER_REDO: a panel that
// passed PROBE_FAST keeps its decision (one round); otherwise its recomputed first round is judged.
// grid = (ceil(r NPROBE / PD_ENTRIES), matrices): a block adds up the chunks of PD_ENTRIES (column, probe) entries, four
// groups of threads a quarter of the chunks each; the last block of a matrix to arrive (os[OS_BARRIER], left at zero)
// adds up the blocks' sums.  (One block per matrix took 81 us at r = 1024: a serial walk over 2.4 MB.)
enum : int { PROBE_CHECK = 0, PROBE_FAST = 1, PROBE_AFTER_REDO = 2 };
constexpr int PD_ENTRIES = 128, PD_GROUPS = 4;
__global__ void __launch_bounds__(PD_ENTRIES * PD_GROUPS) k_probe_decide(const float* __restrict__ part, int chunks, i64 r, int* __restrict__ os,
                                                                         float tau_f, int* __restrict__ rounds_total, float* __restrict__ sums,
                                                                         i64 wstride, int phase) {
  pdl_enter();
  part += (i64)blockIdx.y * wstride; sums += (i64)blockIdx.y * wstride;
  os += (i64)blockIdx.y * OS_SLOT_INTS;
  if (phase == PROBE_AFTER_REDO && os[OS_DONE] != 0) {
    if (threadIdx.x == 0 && blockIdx.x == 0) { os[OS_ROUNDS] = 1; atomicAdd(rounds_total, 1); }
    return;
  }
  __shared__ float red[PD_GROUPS][PD_ENTRIES];
  __shared__ int s_last;
  const int t = threadIdx.x % PD_ENTRIES, grp = threadIdx.x / PD_ENTRIES;
  const i64 x = (i64)blockIdx.x * PD_ENTRIES + t;
  const int per = (chunks + PD_GROUPS - 1) / PD_GROUPS, c0 = grp * per, c1 = min(chunks, c0 + per);
  float w = 0.f;
  if (x < r * NPROBE) {
#pragma unroll 16      // (sixteen chunks' loads in flight; the sum keeps its order)
    for (int c = c0; c < c1; ++c) w += part[(i64)c * r * NPROBE + x];
  }
  red[grp][t] = w;
  __syncthreads();
  if (threadIdx.x < PD_ENTRIES) {
    w = (red[0][t] + red[1][t]) + (red[2][t] + red[3][t]);
    const float dlt = (x < r * NPROBE) ? w - probe_sign(x / NPROBE, (int)(x % NPROBE)) : 0.f;
    red[0][t] = dlt * dlt;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    float e = (red[0][t] + red[0][t + 32]) + (red[0][t + 64] + red[0][t + 96]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (t == 0) {
      sums[blockIdx.x] = e;
      __threadfence();
      s_last = (atomicAdd(&os[OS_BARRIER], 1) == (int)gridDim.x - 1) ? 1 : 0;
    }
  }
  __syncthreads();
  if (s_last == 0 || threadIdx.x >= 32) return;
  __threadfence();
  float e = 0.f;
  for (int c = t; c < (int)gridDim.x; c += 32) e += __ldcg(sums + c);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if (t == 0) {
    os[OS_BARRIER] = 0;
    const float est = e / (float)NPROBE;
    os[OS_MAXDEV] = __float_as_int(est);
    const bool failed = os[OS_FAIL] != 0;       // a pivot of the first round failed: the fallback redoes the panel
    const bool done = !failed && (est <= tau_f * tau_f * (float)r);      // false for NaN
    if (phase == PROBE_FAST) {
      os[OS_DONE] = done ? 1 : 0;
    } else {
      const int extra = (phase == PROBE_AFTER_REDO) ? 1 : 0;
      os[OS_DONE] = (done || failed) ? 1 : 0;
      os[OS_ROUNDS] = (done ? 1 : 2) + extra;
      atomicAdd(rounds_total, (done ? 1 : 2) + extra);
    }
  }
}

// Clears the round state of a step slot (keeps the fail flag): a second orthonormalization in one step.
__global__ void k_reset_rounds(int* __restrict__ os) {
  pdl_enter();
  os += (i64)blockIdx.x * OS_SLOT_INTS;
  os[OS_DONE] = 0; os[OS_GOOD] = 0; os[OS_FLOORED] = 0; os[OS_MAXDEV] = 0; os[OS_ROUNDS] = 0;
}

// After the last adaptive round: a panel that never became well conditioned is
// reported; if pivots were still being raised the step is cancelled (rank-deficient P).
__global__ void k_orth_finish(int* __restrict__ os, int* __restrict__ status) {
  pdl_enter();
  os += (i64)blockIdx.x * OS_SLOT_INTS;
  if (os[OS_DONE] != 0) return;
  if (os[OS_GOOD] == 0 && os[OS_FLOORED] != 0) {
    os[OS_FAIL] = 1;
    atomicOr(status, DION_STATUS_BREAKDOWN);
  } else {
    atomicOr(status, DION_STATUS_ILLCOND);
  }
}

// ---------------------------------------------------------------------------
// Fallback of Cholesky QR, on the device: when a pivot of CholeskyQR2 was not positive (the panel is too
// ill conditioned for the Gram matrix in fp32; the paper falls back to a QR factorization), the panel saved
// before the first round is orthonormalized column by column with classical Gram-Schmidt applied twice
// (the thin-QR factor with positive diagonal, like every other mode), in ONE cooperative launch that returns
// at once when no matrix of the chain failed: no host round trip, no launches beyond this one.
//
// CTA c owns a block of rows of the panel and only ever touches its own rows of U; what crosses CTAs are the
// partial dot products (part[c][k], summed in fixed CTA order into h[k]) and the partial squared norms,
// separated by grid-wide barriers (5 per column).  Column j, pass p: h_k = sum_i U[i][k] U[i][j] for k < j
// (pass 0 also k = j: the squared norm before orthogonalization), U[:, j] -= U[:, <j] h, then the norm and
// the scaling.  A column whose norm falls below CGS_DEFLATE_REL of what it was is linearly dependent on its
// predecessors to fp32 accuracy: the step is cancelled (OS_FAIL, DION_STATUS_BREAKDOWN) as before.
// Every barrier wait is bounded; when one runs out the kernel gives up with DION_STATUS_TIMEOUT and the step
// stays cancelled.
// ---------------------------------------------------------------------------
constexpr float CGS_DEFLATE_REL = 2e-6f;
constexpr int CGS_PASSES = 2;
constexpr int CGS_MAX_ROWS_PER_CTA = 1024;   // floats of shared memory for the CTA's piece of the current column

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Grid-wide barrier on a monotonic arrival counter: barrier number `epoch` (1, 2, ...) is passed when
// epoch * gridDim.x arrivals have been counted.  Returns false when the wait ran out or an earlier one did.
__device__ __forceinline__ bool cgs_grid_barrier(unsigned* counter, unsigned& epoch, long long limit, int* status,
                                                 volatile int* s_dead) {
  __syncthreads();
  ++epoch;
  if (threadIdx.x == 0 && !*s_dead) {
    __threadfence();
    atomicAdd(counter, 1u);
    const unsigned target = epoch * gridDim.x;
    const long long t0 = clock64();
    while (ld_acquire_u32(counter) < target) {
      if (clock64() - t0 > limit) {
        *s_dead = 1;
        atomicOr(status, DION_STATUS_TIMEOUT);
        break;
      }
      __nanosleep(100);
    }
    __threadfence();
  }
  __syncthreads();
  return *s_dead == 0;
}

__device__ __forceinline__ float cgs_block_sum(float v, float* red) {
  const int tid = threadIdx.x;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((tid & 31) == 0) red[tid >> 5] = v;
  __syncthreads();
  float t = 0.f;
  if (tid < 8) t = red[tid];
  if (tid < 32) {
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (tid == 0) red[8] = t;
  }
  __syncthreads();
  const float out = red[8];
  __syncthreads();
  return out;
}

// Pin: the saved panel (rows x r, ld); U: where the orthonormal factor goes (ld).  part: gridDim.x * r floats,
// hvec: r floats, npart: gridDim.x floats -- per matrix, wstride floats apart like every scratch offset.
__global__ void __launch_bounds__(256) k_cgs_fallback(const float* __restrict__ Pin, float* __restrict__ U, i64 ld,
                                                      i64 rows, i64 r, float* __restrict__ part, float* __restrict__ hvec,
                                                      float* __restrict__ npart, int* __restrict__ os_base,
                                                      int* __restrict__ status, int* __restrict__ fallbacks,
                                                      i64 wstride, int nb, long long spin_limit, const float* __restrict__ second) {
  __shared__ float colj[CGS_MAX_ROWS_PER_CTA];
  __shared__ float red[9];
  __shared__ int s_dead;
  __shared__ float s_val;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = (int)gridDim.x, c = (int)blockIdx.x;
  const i64 rpc = (rows + G - 1) / G;
  const i64 i0 = min(rows, (i64)c * rpc), i1 = min(rows, i0 + rpc);
  const int nmy = (int)(i1 - i0);
  {      // nearly always there is nothing to do: all flags at once (one after another 48 matrices were 14 us of a step; twelve blocks of hidden size 768 in one call: 1606 -> 1588 us)
    bool busy = false;
    for (int b = tid; b < nb; b += 256) {
      const int* os = os_base + (i64)b * OS_SLOT_INTS;
      busy = busy || os[OS_FAIL] != 0 || (second != nullptr && os[OS_DONE] == 0);
    }
    if (!__syncthreads_or(busy)) return;
  }
  for (int b = 0; b < nb; ++b) {
    int* os = os_base + (i64)b * OS_SLOT_INTS;
    if (os[OS_FAIL] == 0) {                         // written by an earlier launch: every CTA reads the same value
      if (second != nullptr && os[OS_DONE] == 0) {      // the second round ran: its result to where U is expected
        const float* V = second + (i64)b * wstride;
        float* Ub = U + (i64)b * wstride;
        for (i64 e = (i64)c * 256 + tid; e < rows * r; e += (i64)G * 256) {
          const i64 i = row_of(e, r), k = e - i * r;
          Ub[i * ld + k] = V[i * r + k];
        }
      }
      continue;
    }
    const float* Pb = Pin + (i64)b * wstride;
    float* Ub = U + (i64)b * wstride;
    float* partb = part + (i64)b * wstride;
    float* hb = hvec + (i64)b * wstride;
    float* nb_part = npart + (i64)b * wstride;
    unsigned* counter = reinterpret_cast<unsigned*>(os + OS_BARRIER);
    unsigned epoch = 0;
    if (tid == 0) s_dead = 0;
    __syncthreads();
    bool ok = true, deficient = false;
    for (i64 e = tid; e < (i64)nmy * r; e += 256) {
      const i64 i = i0 + e / r, k = e % r;
      Ub[i * ld + k] = Pb[i * ld + k];
    }
    __syncthreads();
    for (i64 j = 0; j < r && ok && !deficient; ++j) {
      for (int i = tid; i < nmy; i += 256) colj[i] = Ub[(i0 + i) * ld + j];
      __syncthreads();
      float before = 0.f;
      for (int pass = 0; pass < CGS_PASSES && ok; ++pass) {
        const i64 nk = j + (pass == 0 ? 1 : 0);     // pass 0: k = j is the squared norm before orthogonalization
        for (i64 k = tid; k < nk; k += 256) {
          float a0 = 0.f, a1 = 0.f;
          int i = 0;
          for (; i + 1 < nmy; i += 2) {
            a0 = fmaf(Ub[(i0 + i) * ld + k], colj[i], a0);
            a1 = fmaf(Ub[(i0 + i + 1) * ld + k], colj[i + 1], a1);
          }
          if (i < nmy) a0 = fmaf(Ub[(i0 + i) * ld + k], colj[i], a0);
          partb[(i64)c * r + k] = a0 + a1;
        }
        ok = cgs_grid_barrier(counter, epoch, spin_limit, status, &s_dead);
        if (!ok) break;
        {   // fixed-order sums over the CTAs, the k range split over the grid
          const i64 per = (nk + G - 1) / G;
          const i64 k0 = (i64)c * per, k1 = min(nk, k0 + per);
          for (i64 k = k0 + tid; k < k1; k += 256) {
            float sum = 0.f;
            for (int cc = 0; cc < G; ++cc) sum += partb[(i64)cc * r + k];
            hb[k] = sum;
          }
        }
        ok = cgs_grid_barrier(counter, epoch, spin_limit, status, &s_dead);
        if (!ok) break;
        if (pass == 0) before = hb[j];
        if (j > 0) {
          for (int i = warp; i < nmy; i += 8) {       // a warp per row: lanes stride over k
            const float* urow = Ub + (i0 + i) * ld;
            float acc = 0.f;
            for (i64 k = lane; k < j; k += 32) acc = fmaf(urow[k], hb[k], acc);
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
            if (lane == 0) colj[i] -= acc;
          }
          __syncthreads();
        }
      }
      if (!ok) break;
      float sq = 0.f;
      for (int i = tid; i < nmy; i += 256) sq = fmaf(colj[i], colj[i], sq);
      sq = cgs_block_sum(sq, red);
      if (tid == 0) nb_part[c] = sq;
      ok = cgs_grid_barrier(counter, epoch, spin_limit, status, &s_dead);
      if (!ok) break;
      if (tid == 0) {
        float tot = 0.f;
        for (int cc = 0; cc < G; ++cc) tot += nb_part[cc];
        s_val = tot;
      }
      __syncthreads();
      const float after = s_val;
      // every CTA sees the same two sums: the same decision everywhere
      if (!(after > CGS_DEFLATE_REL * CGS_DEFLATE_REL * before) || !(before < __int_as_float(0x7f800000))) {
        deficient = true;
        break;
      }
      const float inv = rsqrtf(after);
      for (int i = tid; i < nmy; i += 256) Ub[(i0 + i) * ld + j] = colj[i] * inv;
      __syncthreads();
    }
    if (c == 0 && tid == 0) {
      if (ok && !deficient) {
        os[OS_FAIL] = 0;
        atomicAdd(fallbacks, 1);
      } else {
        os[OS_FAIL] = 1;
        if (deficient) atomicOr(status, DION_STATUS_BREAKDOWN);
      }
    }
    __syncthreads();
  }
}

// rows x cols from one matrix to another (four elements at a time where both allow it).
__device__ __forceinline__ void copy_rows(const float* __restrict__ src, i64 lds, float* __restrict__ dst, i64 ldd, i64 rows, i64 cols) {
  const i64 stride = (i64)gridDim.x * blockDim.x;
  if (((cols | lds | ldd) & 3) == 0 && (((uintptr_t)src | (uintptr_t)dst) & 15) == 0) {
    const i64 per_row = cols / 4;
    for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < rows * per_row; e += stride) {
      const i64 i = row_of(e, per_row), c = (e - i * per_row) * 4;
      *reinterpret_cast<float4*>(dst + i * ldd + c) = *reinterpret_cast<const float4*>(src + i * lds + c);
    }
    return;
  }
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < rows * cols; e += stride) {
    const i64 i = row_of(e, cols), c = e - i * cols;
    dst[i * ldd + c] = src[i * lds + c];
  }
}

// Copies a rows x cols block between two matrices (leading dimensions lds, ldd).  latch_to (optional): set when *latch_from is (a
// breakdown carried from one call of a multi-call step to the next).
__global__ void k_copy_block(const float* __restrict__ src, i64 lds, float* __restrict__ dst, i64 ldd,
                             i64 rows, i64 cols, const int* __restrict__ skip_flag, i64 wstride,
                             const int* __restrict__ latch_from, int* __restrict__ latch_to, int* __restrict__ slots) {
  pdl_enter();
  clear_slot(slots);
  if (latch_to != nullptr && blockIdx.x == 0 && threadIdx.x == 0 && *latch_from != 0) *latch_to = 1;
  if (skip_flag != nullptr && skip_flag[(i64)blockIdx.y * OS_SLOT_INTS] != 0) return;
  copy_rows(src + (i64)blockIdx.y * wstride, lds, dst + (i64)blockIdx.y * wstride, ldd, rows, cols);     // batched over blockIdx.y
}

// Copies a rows x r panel (ld = ldv) into Q (ld = ldq) unless the step was flagged.
// `only_if` (optional): the copy happens only when (*only_if & only_mask) != 0.
__global__ void k_copy_panel(const float* __restrict__ V, i64 ldv, float* __restrict__ Q, i64 ldq,
                             i64 rows, i64 r, const int* __restrict__ skip_flag,
                             const int* __restrict__ only_if, i64 wstride, int only_mask) {
  pdl_enter();
  V += (i64)blockIdx.y * wstride;                                         // batched over blockIdx.y
  if (wstride != 0) Q += (i64)blockIdx.y * wstride;
  if (skip_flag != nullptr && skip_flag[(i64)blockIdx.y * OS_SLOT_INTS] != 0) return;
  if (only_if != nullptr && (only_if[(i64)blockIdx.y * OS_SLOT_INTS] & only_mask) == 0) return;
  copy_rows(V, ldv, Q, ldq, rows, r);
}

// ---------------------------------------------------------------------------
// Householder QR (unblocked), the slow robust mode.
// ---------------------------------------------------------------------------

// Column j: builds the unit reflector v (stored in V[j:, j]) from A[j:, j] and
// records R_qr[j][j] = alpha in diag[j].  One block of 1024 threads.
__global__ void __launch_bounds__(1024) k_hh_reflector(float* __restrict__ A, i64 lda, i64 m, i64 j,
                                                       float* __restrict__ V, i64 ldv,
                                                       float* __restrict__ diag) {
  __shared__ float red[1024];
  __shared__ float s_alpha, s_vnorm;
  const int tid = threadIdx.x;
  float s = 0.f;
  for (i64 i = j + tid; i < m; i += 1024) { const float v = A[i * lda + j]; s = fmaf(v, v, s); }
  red[tid] = s;
  __syncthreads();
  for (int w = 512; w > 0; w >>= 1) { if (tid < w) red[tid] += red[tid + w]; __syncthreads(); }
  if (tid == 0) {
    const float norm = sqrtf(red[0]);
    const float a0 = A[j * lda + j];
    const float alpha = (a0 >= 0.f) ? -norm : norm;
    // ||x - alpha e1||^2 = 2 norm^2 + 2 norm |x0|
    s_alpha = alpha;
    s_vnorm = sqrtf(2.f * norm * (norm + fabsf(a0)));
    diag[j] = alpha;
  }
  __syncthreads();
  const float alpha = s_alpha, vn = s_vnorm;
  for (i64 i = j + tid; i < m; i += 1024) {
    float v = A[i * lda + j];
    if (i == j) v -= alpha;
    V[i * ldv + j] = (vn > 0.f) ? v / vn : 0.f;
  }
}

// T[j0:, c] -= 2 v (v^T T[j0:, c]) for the columns c in [c_begin, c_end); v = V[j0:, vj].
// grid.x = column chunks of 32; block = 32 x 8 (32 columns, 8 row lanes).
__global__ void __launch_bounds__(256) k_hh_apply(float* __restrict__ T, i64 ldt, i64 m, i64 j0,
                                                  const float* __restrict__ V, i64 ldv, i64 vj,
                                                  i64 c_begin, i64 c_end) {
  __shared__ float red[8][33];
  const int cx = threadIdx.x % 32, ry = threadIdx.x / 32;
  const i64 c = c_begin + (i64)blockIdx.x * 32 + cx;
  const bool ok = c < c_end;
  float s = 0.f;
  if (ok) for (i64 i = j0 + ry; i < m; i += 8) s = fmaf(V[i * ldv + vj], T[i * ldt + c], s);
  red[ry][cx] = s;
  __syncthreads();
  float w = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) w += red[k][cx];
  w *= 2.f;
  if (ok) for (i64 i = j0 + ry; i < m; i += 8) T[i * ldt + c] = fmaf(-V[i * ldv + vj], w, T[i * ldt + c]);
}

// U = first r columns of the identity.
__global__ void k_set_identity(float* __restrict__ U, i64 ld, i64 m, i64 r) {
  const i64 total = m * r;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    const i64 i = row_of(e, r), c = e - i * r;
    U[i * ld + c] = (i == c) ? 1.f : 0.f;
  }
}

// Sign convention: negate column j of U wherever diag[j] (= R_qr[j][j]) < 0.
__global__ void k_sign_fix(float* __restrict__ U, i64 ld, i64 m, i64 r, const float* __restrict__ diag) {
  const i64 total = m * r;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    const i64 i = row_of(e, r), c = e - i * r;
    if (diag[c] < 0.f) U[i * ld + c] = -U[i * ld + c];
  }
}

}  // namespace dion
