// The Cholesky factorization of a Gram matrix, the inverse of its factor and the triangular solve of a panel, as ONE
// launch of cooperating CTAs (data flow between 64 x 64 tiles instead of one launch per block column).
#pragma once

#include <stddef.h>

#include "dion_common.cuh"

namespace dion {

// ---------------------------------------------------------------------------------------------------------------
// fp32 products on the warp-level tensor path: x = h + m + l with h, m, l bf16 (8 + 8 + 8 significant bits, every
// remainder rounded to nearest), six of the nine cross products (those dropped are below 2^-26 of the product).  The
// h h terms go to one accumulator, the rest to a second one that is added at the end: one truncating add per K step
// on the main sum.  As accurate as a chain of fp32 FMAs, at 1.3 times their rate -- and, what counts here, an
// operand fragment of a 16 x 8 tile is a few words per lane: a shared-memory load returns at most 128 bytes a cycle
// to the registers of an SM, broadcast or not, which held a 64^3 product with 4 x 4 outputs per thread at 3900 cycles.
// ---------------------------------------------------------------------------------------------------------------
struct Bf3 { uint32_t h, m, l; };      // a pair of neighbouring k (the even one in the low half)

__device__ __forceinline__ Bf3 split3(float x, float y) {
  Bf3 r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r.h) : "f"(y), "f"(x));
  x -= __uint_as_float(r.h << 16); y -= __uint_as_float(r.h & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r.m) : "f"(y), "f"(x));
  x -= __uint_as_float(r.m << 16); y -= __uint_as_float(r.m & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r.l) : "f"(y), "f"(x));
  return r;
}
__device__ __forceinline__ Bf3 split3(float2 v) { return split3(v.x, v.y); }
__device__ __forceinline__ void mma_k16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// acc[i] += A B_i of N 16 x 8 tiles with K = 8: the two halves of a K = 16 mma take two cross products (an m16n8k8 mma
// takes longer than an m16n8k16 one here).  Term by term over the tiles: it is tens of cycles to the next mma on the
// same accumulator.
template <int N>
__device__ __forceinline__ void mma3_k8(float (*acc)[4], const Bf3& a0, const Bf3& a1, const Bf3 (&b)[N]) {
  float s[N][4];
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) s[i][e] = 0.f;
#pragma unroll
  for (int i = 0; i < N; ++i) mma_k16(s[i], a0.l, a1.l, a0.h, a1.h, b[i].h, b[i].l);
#pragma unroll
  for (int i = 0; i < N; ++i) mma_k16(acc[i], a0.m, a1.m, a0.h, a1.h, b[i].m, b[i].h);
#pragma unroll
  for (int i = 0; i < N; ++i) mma_k16(s[i], a0.m, a1.m, a0.h, a1.h, b[i].h, b[i].m);
#pragma unroll
  for (int i = 0; i < N; ++i)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[i][e] += s[i][e];
}

constexpr int CB = 64;      // tile
constexpr int CLD = 72;     // row stride of a tile in shared memory (= 8 mod 32: the fragment loads are free of bank conflicts)
typedef float (*ctile_t)[CLD];

// A 64 x 64 tile over eight warps: warp w holds rows 16 (w / 2) .. + 15 and the 8-column groups 2 j + (w & 1), j = 0 .. 3;
// lane (g, t) = (lane / 4, lane % 4) holds of group j: v[j][0], v[j][1] at row g, columns 2 t, 2 t + 1, v[j][2], v[j][3] at row g + 8.
struct TileLane {
  int row, col;      // of v[0][0]
  __device__ __forceinline__ TileLane(int tid) : row(16 * (tid >> 6) + ((tid & 31) >> 2)), col(8 * ((tid >> 5) & 1) + 2 * (tid & 3)) {}
  __device__ __forceinline__ int r(int e) const { return row + ((e & 2) ? 8 : 0); }
  __device__ __forceinline__ int c(int j, int e) const { return col + 16 * j + (e & 1); }
};

// v = A B^T of 64 x 64 tiles in shared memory (k contiguous in both).  TRI: B is lower triangular (its zeros above the
// diagonal are stored): column c needs k <= c only.  LOWER: only the groups that reach the diagonal or lie below it.
enum : int { MM_FULL = 0, MM_TRI = 1, MM_LOWER = 2 };
__device__ __forceinline__ void tile_nt(ctile_t A, ctile_t B, int mode, int tid, float (&v)[4][4]) {
  const int warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3, rt = warp >> 1, par = warp & 1;
  float s[4][4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) v[j][e] = s[j][e] = 0.f;
  const float* pa = &A[16 * rt + g][2 * t];
  const float* pb = &B[8 * par + g][2 * t];
#pragma unroll 2      // (short on purpose: code that runs once costs more to fetch than to execute)
  for (int kk = 0; kk < CB; kk += 16) {
    float2 fa[4], fb[4][2];
    fa[0] = *reinterpret_cast<const float2*>(pa); fa[1] = *reinterpret_cast<const float2*>(pa + 8 * CLD);
    fa[2] = *reinterpret_cast<const float2*>(pa + 8); fa[3] = *reinterpret_cast<const float2*>(pa + 8 * CLD + 8);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float* q = pb + 16 * j * CLD;
      fb[j][0] = *reinterpret_cast<const float2*>(q);
      fb[j][1] = *reinterpret_cast<const float2*>(q + 8);
    }
    const Bf3 a0 = split3(fa[0]), a1 = split3(fa[1]), a2 = split3(fa[2]), a3 = split3(fa[3]);
    // (two column groups at a time, term by term: it is tens of cycles to the next mma on the same accumulator)
#pragma unroll
    for (int j0 = 0; j0 < 4; j0 += 2) {
      // (one group decides for both: the other one's operands are zero, or its entries unused)
      if (mode == MM_TRI && kk > 8 * (2 * (j0 + 1) + par) + 7) continue;      // (uniform)
      if (mode == MM_LOWER && 2 * j0 + par > 2 * rt + 1) continue;
      Bf3 b[2][2];
#pragma unroll
      for (int i = 0; i < 2; ++i) { b[i][0] = split3(fb[j0 + i][0]); b[i][1] = split3(fb[j0 + i][1]); }
#pragma unroll
      for (int i = 0; i < 2; ++i) mma_k16(s[j0 + i], a0.l, a1.l, a2.l, a3.l, b[i][0].h, b[i][1].h);
#pragma unroll
      for (int i = 0; i < 2; ++i) mma_k16(v[j0 + i], a0.h, a1.h, a2.h, a3.h, b[i][0].h, b[i][1].h);
#pragma unroll
      for (int i = 0; i < 2; ++i) mma_k16(s[j0 + i], a0.h, a1.h, a2.h, a3.h, b[i][0].l, b[i][1].l);
#pragma unroll
      for (int i = 0; i < 2; ++i) mma_k16(s[j0 + i], a0.m, a1.m, a2.m, a3.m, b[i][0].m, b[i][1].m);
#pragma unroll
      for (int i = 0; i < 2; ++i) mma_k16(s[j0 + i], a0.m, a1.m, a2.m, a3.m, b[i][0].h, b[i][1].h);
#pragma unroll
      for (int i = 0; i < 2; ++i) mma_k16(s[j0 + i], a0.h, a1.h, a2.h, a3.h, b[i][0].m, b[i][1].m);
    }
    pa += 16;
    pb += 16;
  }
#pragma unroll
  for (int j = 0; j < 4; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) v[j][e] += s[j][e];
}
// tile in shared memory from the lanes' entries
__device__ __forceinline__ void tile_put(ctile_t T, const TileLane& l, const float (&v)[4][4]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    *reinterpret_cast<float2*>(&T[l.row][l.col + 16 * j]) = make_float2(v[j][0], v[j][1]);
    *reinterpret_cast<float2*>(&T[l.row + 8][l.col + 16 * j]) = make_float2(v[j][2], v[j][3]);
  }
}

__device__ __forceinline__ void tile_get(ctile_t T, const TileLane& l, float (&v)[4][4]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float2 a = *reinterpret_cast<const float2*>(&T[l.row][l.col + 16 * j]), b = *reinterpret_cast<const float2*>(&T[l.row + 8][l.col + 16 * j]);
    v[j][0] = a.x; v[j][1] = a.y; v[j][2] = b.x; v[j][3] = b.y;
  }
}

// ---------------------------------------------------------------------------------------------------------------
// Cholesky factor and inverse of one 64 x 64 block by 256 threads, both in shared memory.
//
// Bound by the serial chain of 64 pivots.  The block is factored in panels of eight columns:
//   warps 0-1 (the chain): a thread owns a row, its eight panel entries in registers, and ALL of them factor the 8 x 8
//     diagonal piece redundantly in registers, so that inside a panel nothing crosses threads: a column costs the
//     pivot's reciprocal square root and three dependent operations (~45 cycles), and the rows below are solved in the
//     issue slots between them.
//   warps 4-7: warp 4 + w keeps rows 16 w .. 16 w + 15 of the columns that are still to come in registers (16 x 8
//     tiles of the tensor path), takes off every finished panel (rank 8) -- the next panel's columns first, which go back
//     to shared memory for the chain -- and uses a column tile that has been handed over for the terms of the inverse,
//     S = sum L X.
//   warps 2-3 (the inverse X): one column per thread; with S of a panel's rows in place, an 8 x 8 substitution.
// Everything is a short loop over the panels: the code is fetched once.
// (One thread factoring the piece, three barriers per panel, FMA updates and the inverse by doubling took 23 k cycles.)
//
// L: the scaled block on entry (lower triangle; identity padding beyond a ragged block), the scaled factor on return
// (entries above the diagonal are not meaningful).  X: the inverse on return (lower, zeros above; zero rows for deflated
// columns).  Named barriers 1 (256
// threads), 2 and 3 (192).
// Pivot rules: see k_chol_flow.
// ---------------------------------------------------------------------------------------------------------------
template <int ID, int N>
__device__ __forceinline__ void bar_named() { asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(N) : "memory"); }

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ void st4(float* p, float4 v) { *reinterpret_cast<float4*>(p) = v; }
__device__ __forceinline__ void ld8(float (&v)[8], const float* p) {
  const float4 a = ld4(p), b = ld4(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void st8(float* p, const float (&v)[8]) {
  st4(p, make_float4(v[0], v[1], v[2], v[3]));
  st4(p + 4, make_float4(v[4], v[5], v[6], v[7]));
}

// What potrf64 needs to know of a block's pivots (shared memory), written by one warp (potrf64_setup).
struct alignas(16) Potrf64Set {
  float gd[CB];          // reference values of the pivots, scaled by s2
  float floor[CB];       // smallest pivots taken as they are
  float alt_inv[CB];     // what stands in for 1 / L[j][j] of a smaller one
  float s2, s1;          // the block's scale and its root
};
struct alignas(16) Potrf64Aux {
  float dg[2][64];       // the diagonal piece of a panel, by parity
  float rdiag[CB];       // 1 / L[j][j]
  unsigned bad8[8];      // per panel: the columns whose pivot was replaced
};
static_assert(offsetof(Potrf64Set, floor) % 16 == 0 && offsetof(Potrf64Set, alt_inv) % 16 == 0 && sizeof(Potrf64Set) % 16 == 0 &&
              offsetof(Potrf64Aux, rdiag) % 16 == 0, "read and written 16 bytes at a time");

// g0, g1: the reference values of columns lane and lane + 32.  s2 is the power of four by which the block has to be
// multiplied when it is put into L, so that its pivots are far from the subnormal range (the reciprocal square root
// below flushes that to zero); the factor comes out scaled by its root s1, the inverse unscaled.
__device__ __forceinline__ void potrf64_setup(Potrf64Set& st, float g0, float g1, float floor_rel, int lane) {
  const float inf = __int_as_float(0x7f800000);
  const float m = __uint_as_float(__reduce_max_sync(0xffffffffu, max(__float_as_uint(fabsf(g0)), __float_as_uint(fabsf(g1)))));
  int e = ((int)(__float_as_uint(m) >> 23) - 127) & ~1;      // m in [2^e, 2^(e + 2))
  if (!(m < inf) || m == 0.f) e = 0;
  e = max(-126, min(126, e));
  const float s2 = __uint_as_float((unsigned)(127 - e) << 23), s1 = __uint_as_float((unsigned)(127 - e / 2) << 23);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float g = (h ? g1 : g0) * s2;
    const float fl = floor_rel * g;
    // Zero or non-finite column: unit pivot, of the block as it was before the scale.  (A column whose entries are beyond the
    // panel's pair has a zero here; it comes back in a later round only if nothing divides it by the others' norm.)
    const float alt = (fl > 0.f && fl < inf) ? fl : s2;
    st.gd[lane + 32 * h] = g;
    st.floor[lane + 32 * h] = fl;
    st.alt_inv[lane + 32 * h] = rsqrtf(alt);
  }
  if (lane == 0) { st.s2 = s2; st.s1 = s1; }
}

// Dg, DPg (optional): the inverse also goes to global memory, dense, DPg with the rows of deflated columns zeroed (as X in
// shared memory); both complete behind the last barrier.
__device__ __forceinline__ void potrf64(ctile_t L, ctile_t X, const Potrf64Set& set, Potrf64Aux& aux, float floor_rel,
                                        int* __restrict__ os, int* __restrict__ status, int tid, float* __restrict__ Dg = nullptr,
                                        float* __restrict__ DPg = nullptr) {
  constexpr int W = 8, NPAN = CB / W;
  const float inf = __int_as_float(0x7f800000);
  if (tid < 64) {
    // ---------------------------------------------------------------- the chain: one row each
    // (No divergent branch and no branch on data between the barriers: a shared-memory load takes a warp 5 to 8 cycles
    // to issue and a branch cuts the schedule; entries above the diagonal are written along.)
    const int i = tid, warp = tid >> 5;
    unsigned long long bad = 0;      // columns whose pivot was replaced
    float fl[W], alt[W];
    ld8(fl, &set.floor[0]);
    ld8(alt, &set.alt_inv[0]);
    const float bad_scale = (floor_rel > 0.f) ? 0.f : 1.f;
    if (i < W) {
      float a[W];
      ld8(a, &L[i][0]);
      st8(&aux.dg[0][i * W], a);
    }
    bar_named<4, 64>();
#pragma unroll 1
    for (int p = 0; p < NPAN; ++p) {
      const int c0 = W * p;
      if (c0 < 32 * (warp + 1)) {      // (rows of this warp at or below the piece)
        float d[W][W], inv[W], a[W];
        unsigned b8 = 0;
        const float* dg = aux.dg[p & 1];
#pragma unroll
        for (int q = 0; q < W; ++q) {
          const float4 u = ld4(dg + q * W);
          d[q][0] = u.x; d[q][1] = u.y; d[q][2] = u.z; d[q][3] = u.w;
          if (q >= 4) {
            const float4 v = ld4(dg + q * W + 4);
            d[q][4] = v.x; d[q][5] = v.y; d[q][6] = v.z; d[q][7] = v.w;
          }
        }
        ld8(a, &L[i][c0]);
#pragma unroll
        for (int j = 0; j < W; ++j) {
          const float pv = d[j][j];
          const bool good = (pv > fl[j]) & (pv < inf);
          float iv;
          asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(iv) : "f"(pv));
          const float sc = good ? iv : bad_scale;
          inv[j] = good ? iv : alt[j];
          d[j][j] = good ? pv * iv : 1.f;
          b8 |= good ? 0u : (1u << j);
#pragma unroll
          for (int q = j + 1; q < W; ++q) d[q][j] *= sc;
          a[j] *= sc;
#pragma unroll
          for (int c = j + 1; c < W; ++c) {
#pragma unroll
            for (int q = c; q < W; ++q) d[q][c] = fmaf(-d[q][j], d[c][j], d[q][c]);
            a[c] = fmaf(-a[j], d[c][j], a[c]);
          }
        }
        const int r = i - c0;
#pragma unroll
        for (int c = 0; c < W; ++c) a[c] = (c == r) ? d[c][c] : a[c];
        st8(&L[i][c0], a);
        st8(&aux.rdiag[c0], inv);      // (every lane the same)
        aux.bad8[p] = b8;
        bad |= (unsigned long long)b8 << c0;
      }
      bar_named<1, 256>();      // panel p is final
      if (p + 1 < NPAN) {
        ld8(fl, &set.floor[c0 + W]);
        ld8(alt, &set.alt_inv[c0 + W]);
        bar_named<2, 192>();      // the next panel's columns are up to date
      }
    }
    if (warp == 1 && bad != 0) {
      if (tid == 32) {
        if (floor_rel > 0.f) {
          atomicAdd(&os[OS_FLOORED], __popcll(bad));
        } else {
          os[OS_FAIL] = 1;
          if (status != nullptr) atomicOr(status, DION_STATUS_BREAKDOWN);   // nullptr: a fallback follows in the same step
        }
      }
    }
    if (warp == 1 && floor_rel > 0.f) {      // smallest pivot relative to its column's squared norm (deflated columns apart)
      const int lane = tid & 31;
      float m = inf;
#pragma unroll
      for (int h = 0; h < CB; h += 32) {
        const int j = lane + h;
        const float l = L[j][j];
        if (((bad >> j) & 1) == 0) m = fminf(m, __fdividef(l * l, set.gd[j]));
      }
      const unsigned u = __reduce_min_sync(0xffffffffu, __float_as_uint(m));      // (all are >= 0: ordered like their bits)
      if (lane == 0) atomicMin(&os[OS_MINREL], (int)u);
    }
  } else if (tid < 128) {
    // ---------------------------------------------------------------- the inverse: one column each
    const int col = tid - 64;
    const float xscale = set.s1;
#pragma unroll 1
    for (int p = 0; p < NPAN; ++p) {
      const int c0 = W * p;
      bar_named<1, 256>();      // panel p is final, S of its rows is in X's place (columns < c0)
      // X[c0 + r][col] = (e - S - sum_{q<r} L x_q) / L_rr, column by column of the 8 x 8 piece
      float x[W], rd[W], l[W][W];
#pragma unroll
      for (int r = 0; r < W; ++r) x[r] = X[c0 + r][col];
#pragma unroll
      for (int r = 0; r < W; ++r) {
        const float4 u = ld4(&L[c0 + r][c0]);
        l[r][0] = u.x; l[r][1] = u.y; l[r][2] = u.z; l[r][3] = u.w;
        if (r > 4) {
          const float4 v = ld4(&L[c0 + r][c0 + 4]);
          l[r][4] = v.x; l[r][5] = v.y; l[r][6] = v.z; l[r][7] = v.w;
        }
      }
      ld8(rd, &aux.rdiag[c0]);
#pragma unroll
      for (int r = 0; r < W; ++r) x[r] = (col < c0) ? -x[r] : ((c0 + r == col) ? xscale : 0.f);
#pragma unroll
      for (int r = 0; r < W; ++r) {
        x[r] *= rd[r];
#pragma unroll
        for (int q = r + 1; q < W; ++q) x[q] = fmaf(-l[q][r], x[r], x[q]);
      }
      if (Dg != nullptr) {
#pragma unroll
        for (int r = 0; r < W; ++r) Dg[(c0 + r) * CB + col] = x[r];
      }
      if (floor_rel > 0.f) {
        // the row of a deflated column (whose entries of L below the diagonal are zero: no other row of X takes it up)
        const unsigned b8 = aux.bad8[p];
#pragma unroll
        for (int r = 0; r < W; ++r) x[r] = ((b8 >> r) & 1) ? 0.f : x[r];
        if (DPg != nullptr) {
#pragma unroll
          for (int r = 0; r < W; ++r) DPg[(c0 + r) * CB + col] = x[r];
        }
      }
#pragma unroll
      for (int r = 0; r < W; ++r) X[c0 + r][col] = x[r];
      if (p + 1 < NPAN) bar_named<3, 192>();
    }
  } else {
    // ---------------------------------------------------------------- columns to come, then terms of the inverse
    const int w = (tid - 128) >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
    const int row = 16 * w + g;
    // slot i of panel p: column tile C = p + 1 + i (mod 8): minus the block's entries until they are handed over (slot 0),
    // then, from the last slot on, the tile's terms of S
    float acc[NPAN][4];
#pragma unroll
    for (int i = 0; i < NPAN; ++i)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][e] = (i == NPAN - 1) ? 0.f : -L[row + ((e & 2) ? 8 : 0)][8 * (i + 1) + 2 * t + (e & 1)];
#pragma unroll 1
    for (int p = 0; p < NPAN; ++p) {
      const int c0 = W * p, c1 = c0 + W;
      bar_named<1, 256>();      // panel p is final
      if (p + 1 == NPAN) break;
      if (16 * w + 15 < c1) {      // (no rows of this warp are left)
        bar_named<2, 192>();
        bar_named<3, 192>();
        continue;
      }
      const float2 f0 = *reinterpret_cast<const float2*>(&L[row][c0 + 2 * t]), f1 = *reinterpret_cast<const float2*>(&L[row + 8][c0 + 2 * t]);
      const float2 fb = *reinterpret_cast<const float2*>(&L[c1 + g][c0 + 2 * t]);
      const Bf3 a0 = split3(f0), a1 = split3(f1);
      {      // the next panel's columns first: the chain waits for them
        const Bf3 b[1] = {split3(fb)};
        mma3_k8<1>(acc, a0, a1, b);
        const float2 o0 = make_float2(-acc[0][0], -acc[0][1]), o1 = make_float2(-acc[0][2], -acc[0][3]);
        *reinterpret_cast<float2*>(&L[row][c1 + 2 * t]) = o0;
        *reinterpret_cast<float2*>(&L[row + 8][c1 + 2 * t]) = o1;
        if (w == c1 >> 4) *reinterpret_cast<float2*>(&aux.dg[(p + 1) & 1][g * W + 2 * t]) = (c1 & 8) ? o1 : o0;
      }
      bar_named<2, 192>();
#pragma unroll
      for (int i = 0; i < NPAN; ++i)
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[i][e] = (i + 1 < NPAN) ? acc[(i + 1) % NPAN][e] : 0.f;
      bar_named<3, 192>();      // X's rows of panel p are there
      // now slot i: C = p + 2 + i (mod 8), i < 7: the columns to come take off L L^T, the others add L X; then S of the tile
      // handed over at panel p - 1 (slot 6) and, from the next panel on, the one handed over now (slot 7)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        Bf3 b[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int C = p + 2 + 4 * h + i;
          const float* q = (C >= NPAN) ? &X[c0 + 2 * t][8 * (C - NPAN) + g] : &L[8 * C + g][c0 + 2 * t];
          float x = 0.f, y = 0.f;
          if (4 * h + i < NPAN - 1) { x = q[0]; y = q[(C >= NPAN) ? CLD : 1]; }
          b[i] = split3(x, y);
        }
        if (h == 0) mma3_k8<4>(acc, a0, a1, b);
        else {
          const Bf3 b3[3] = {b[0], b[1], b[2]};
          mma3_k8<3>(acc + 4, a0, a1, b3);
        }
      }
      if (w == c1 >> 4) {      // S of the next panel's rows: column tiles 0 .. p sit in slots 6 - p .. 6
        const bool hi = (c1 & 8) != 0;
#pragma unroll
        for (int i = 0; i < NPAN - 1; ++i) {
          const int C = p + 2 + i - NPAN;
          if (C >= 0) *reinterpret_cast<float2*>(&X[c1 + g][8 * C + 2 * t]) = hi ? make_float2(acc[i][2], acc[i][3]) : make_float2(acc[i][0], acc[i][1]);
        }
      }
    }
  }
  bar_named<1, 256>();
}

// ---------------------------------------------------------------------------------------------------------------
// k_chol_flow: for every matrix b of a chain, on the diagonal square [o, o + sz) of its Gram matrix A (r x r, lower):
//   L L^T = A (lower factor, below the block diagonal), D_k = L_kk^-1, and behind it, tile by tile
//   and beside the rest of the factorization, either
//     solve:    U = P L^-T for a panel P (rows x sz), or
//     inverse:  L^-T of the square (row-major, upper triangular; zeros below the diagonal, of the whole Gram matrix as far as a
//               product of 256-column tiles reads, of a smaller square everywhere) for a solve by tensor-core products, and
//               its largest entry.
// Pivots: with floor_rel == 0 a pivot that is <= 0 or not finite sets os[OS_FAIL] (and DION_STATUS_BREAKDOWN unless
// `status` is null) and is replaced by 1, so that everything downstream stays finite.  With floor_rel > 0 (adaptive
// rounds) a pivot below floor_rel times the column's entry of diag(A) is below the rounding noise of the Gram matrix:
// the column is deflated -- its diagonal entry becomes sqrt(floor), the entries below it zero -- so that the noisy
// column never reaches the trailing matrix and the factor stays nonsingular; a later round finishes the job.
// A diagonal entry of A that is not finite means a NaN or Inf in M, G or Q: os[OS_FAIL] and DION_STATUS_NONFINITE.
//
// The right-looking form took one launch per 64 columns, ~21 us each, whatever the trailing work (r = 1024: 19 launches, 440 us
// with the solve's products; now 160 us and one product).  Bound by the chain of diagonal blocks, ~8.5 us each: under ncu at
// r = 1024 160 us at 1.85 GHz, 9 % of the SMs' issue slots, 0.4 % of DRAM, 18.5 of a warp's 25 cycles per instruction at barriers
// (the runner's service warps, and helpers without a task).  Here the chain
// D_k -> L_{k+1,k} -> A_{k+1,k+1} -> D_{k+1} stays inside ONE CTA (the "runner" of its matrix: two 64^3 products
// and potrf64 per step), and every other tile is a task of a helper CTA, left-looking:
//   L(i,k)    = (A_ik - sum_{j<k} L_ij L_kj^T) D_k^T                       i >= k + 3  (the runner makes i = k + 1)
//   DIAG(k)   = A_kk - sum_{j<k-1} L_kj L_kj^T     for the runner's step k (it adds the last term); also makes L_{k,k-2}
//   SUB(k)    = A_{k,k-1} - sum_{j<k-1} L_kj L_{k-1,j}^T     for the runner's step k; makes L_{k,k-2} for itself: fetched from
//               DIAG it would come one trip through memory later on the chain's second loop, D_{k-2} -> L_{k,k-2} -> step k
//   PANEL(I,k)= (P_Ik - sum_{j<k} U_Ij L_kj^T) D_k^T       64 panel rows (inverse: P = I, the sum starts at j = I)
// A tile's terms are added as soon as their factors exist (double-buffered cp.async), in the order of j whoever runs
// the task: the result does not depend on the schedule.  Progress is published as one counter per row of L and U
// (tiles of a row are finished in the order of k) and one for D; a consumer's thread 0 polls with acquire loads.
// Helper tasks are handed out in the order of steps (the panel's a few steps behind the factor's), so a task only
// ever waits for tasks handed out before it and for the runners, which are resident: the launch is cooperative.  Only the
// preparations are handed out `ahead` steps early; they hold no more than half of the helpers.  Every wait has a cycle limit (then DION_STATUS_TIMEOUT and os[OS_FAIL], and every CTA leaves).
// The last CTA to leave clears the counters for the next launch and evaluates the round (adaptive rounds).
// ---------------------------------------------------------------------------------------------------------------
enum : int { FLOW_TICKET = 0, FLOW_LEFT = 1, FLOW_ABORT = 2, FLOW_SM_BITS = 8, FLOW_SM_WORDS = 8, FLOW_HEAD_INTS = 32 };   // head of the control block
constexpr int FLOW_CTL_INTS = 64 * 1024;      // ints of a context's control block (zero between launches)
constexpr int FLOW_COMPUTE = 256;            // threads that compute ...
constexpr int FLOW_SERVICE = 128;            // ... and the service warps of a runner (four: nothing else fits beside eight anyway)
constexpr int FLOW_THREADS = FLOW_COMPUTE + FLOW_SERVICE;
constexpr int FLOW_IZ = 4;                    // the inverse's rows are stored (as zeros below the diagonal) up to a multiple of this many tiles
// rows of tiles of column k of the inverse that are written (whole: of a square whose largest entry is looked for afterwards)
__host__ __device__ __forceinline__ int flow_inverse_rows(int T, int k, bool whole) {
  const int n = k / FLOW_IZ * FLOW_IZ + FLOW_IZ;
  return (whole || n > T) ? T : n;
}
constexpr int FLOW_LAG = 2;                   // steps by which the panel's tasks follow the factor's

struct FlowArgs {
  const float* A;           // Gram matrix of matrix 0, leading dimension r
  float* L;                 // its factor below the block diagonal (and the runner's prepared tiles); another r x r buffer
  const float* part;        // != null: the Gram matrix is, instead of A, alpha * sum of nsplit partial sums, r x r each (split-K product)
  int nsplit;
  const float* alpha_dev;   // scale of the partial sums (a power of two; alpha_stride apart per matrix), or null
  i64 alpha_stride;
  float* Dinv;              // (r / 64) tiles: D_k; DinvP: D_k with the rows of deflated columns zeroed (may equal Dinv when floor_rel == 0)
  float* DinvP;
  float* gdiag;             // r floats: diag of the whole Gram matrix, from the caller when gdiag_given (a later square of several), else written here
  int gdiag_given;
  const float* Pin;         // solve: panel rows x r (columns of the square start at o), else null
  float* Pout;              // solve: the panel's result; inverse: L^-T in the place of the square (leading dimension r)
  float* xmax;              // inverse: its largest magnitude, wstride apart per matrix (or null)
  i64 rows;                 // panel rows
  i64 r, o, sz;
  float floor_rel;
  int* os; int skips;
  int* status;              // BREAKDOWN goes here (null: quiet), the rest to status_always
  int* status_always;
  int* ctl; int ctl_stride; // control block; ints per matrix after its head
  i64 wstride; int nb;
  int ahead;                // steps by which the preparations are handed out early (they take on every term since the first column)
  int exclusive;            // a runner has its SM to itself: the helper beside it leaves
  int near;                 // a matrix whose OS_GOOD is 2 is left alone too (k_near_identity has formed its factor)
  int round_end;            // evaluate the adaptive round
  float good_rel, done_rel;
  int* rounds_total;
  long long limit;
};

// End of an adaptive round (one thread).  `minrel`, the smallest pivot relative to its column's squared norm, estimates
// 1 / cond^2 of the round's input panel.
//   - no pivot raised and minrel >= done_rel: the input was already orthonormal to ~(1 - done_rel), so this round's
//     output is orthonormal to rounding level: done;
//   - no pivot raised and minrel >= good_rel: cond <~ 1 / sqrt(good_rel); one more round brings orthonormality to
//     rounding level (the CholeskyQR2 argument), after which the remaining rounds are skipped.
__device__ __forceinline__ void round_evaluate(int* __restrict__ os, float good_rel, float done_rel, int* __restrict__ rounds_total) {
  volatile int* v = os;
  v[OS_ROUNDS] = v[OS_ROUNDS] + 1;
  atomicAdd(rounds_total, 1);
  if (v[OS_GOOD] != 0) { v[OS_DONE] = 1; return; }
  const float minrel = __int_as_float(v[OS_MINREL]);
  if (v[OS_FLOORED] == 0) {
    if (minrel >= done_rel) v[OS_DONE] = 1;
    else if (minrel >= good_rel) v[OS_GOOD] = 1;
  }
}

struct FlowTask { int type, b, i, k; };
enum : int { FT_L = 0, FT_SUB = 1, FT_DIAG = 2, FT_PANEL = 3, FT_NONE = 4 };

__device__ __forceinline__ int flow_ld(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void flow_publish(int* p, int v) {     // the CTA's writes before the last barrier come first
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  asm volatile("st.relaxed.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ unsigned flow_smid() {
  unsigned r;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(r));
  return min(r, (unsigned)(32 * FLOW_SM_WORDS - 1));
}
// thread 0: waits until *p >= want; returns the value seen, or -1 when the wait ran out (or another CTA's did)
__device__ __forceinline__ int flow_wait(const int* p, int want, const FlowArgs& f) {
  int v = flow_ld(p);
  if (v >= want) return v;
  const long long t0 = clock64();
  unsigned polls = 0;
  while (true) {
    v = flow_ld(p);
    if (v >= want) return v;
    if ((++polls & 15u) == 0) {
      if (flow_ld(f.ctl + FLOW_ABORT) != 0) return -1;
      if (clock64() - t0 > f.limit) {
        atomicExch(f.ctl + FLOW_ABORT, 1);
        atomicOr(f.status_always, DION_STATUS_TIMEOUT);
        return -1;
      }
    }
  }
}

// rows x cols (<= 64 x 64) of src into a tile, zeros elsewhere.  VEC: 16-byte aligned rows, cols a multiple of 4:
// asynchronous (cp.async, the caller waits); else plain loads.  Reads go to L2: other CTAs have written the data.
template <bool VEC, int NT = FLOW_COMPUTE>
__device__ __forceinline__ void flow_load(ctile_t T, const float* __restrict__ src, i64 ld, int rows, int cols, int tid) {
  if (VEC) {
#pragma unroll 4
    for (int e = tid; e < CB * CB / 4; e += NT) {
      const int i = e >> 4, c = (e & 15) * 4;
      const bool ok = i < rows && c < cols;
      const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&T[i][c]);
      const float* g = ok ? src + (i64)i * ld + c : src;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(g), "r"(ok ? 16 : 0) : "memory");
    }
  } else {
#pragma unroll 8
    for (int e = tid; e < CB * CB; e += NT) {
      const int i = e >> 6, c = e & 63;
      T[i][c] = (i < rows && c < cols) ? __ldcg(src + (i64)i * ld + c) : 0.f;
    }
  }
}
__device__ __forceinline__ void flow_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void flow_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

constexpr int FLOW_SMEM = 6 * CB * CLD * (int)sizeof(float);

template <bool VEC>
__global__ void __launch_bounds__(FLOW_THREADS, 1) k_chol_flow(const __grid_constant__ FlowArgs f) {
  pdl_enter();
  auto skipped = [&](int b) -> bool {
    const int* os = f.os + (i64)b * OS_SLOT_INTS;
    return (f.skips && os[OS_DONE] != 0) || (f.near && os[OS_GOOD] == 2);
  };
  if ((f.skips || f.near) && __syncthreads_and((int)threadIdx.x >= f.nb || skipped((int)threadIdx.x))) return;      // (nb <= 64)
  extern __shared__ __align__(16) float flow_smem[];
  ctile_t SA[2] = {reinterpret_cast<ctile_t>(flow_smem), reinterpret_cast<ctile_t>(flow_smem + 2 * CB * CLD)};
  ctile_t SB[2] = {reinterpret_cast<ctile_t>(flow_smem + CB * CLD), reinterpret_cast<ctile_t>(flow_smem + 3 * CB * CLD)};
  ctile_t SC[2] = {reinterpret_cast<ctile_t>(flow_smem + 4 * CB * CLD), reinterpret_cast<ctile_t>(flow_smem + 5 * CB * CLD)};
  __shared__ Potrf64Set s_set[2];
  __shared__ Potrf64Aux aux;
  __shared__ float s_diag[2][CB];
  __shared__ int s_ready[2];
  __shared__ int s_ok, s_prep;
  __shared__ FlowTask s_task;
  const int tid = threadIdx.x;
  const TileLane tl(tid);      // this thread's 16 entries of a tile
  const int T = (int)((f.sz + CB - 1) / CB);
  const bool solve = f.Pin != nullptr;
  const int NR = solve ? (int)((f.rows + CB - 1) / CB) : 0;      // row blocks of the panel
  const i64 ld = f.r;
  auto cols_of = [&](int k) { return (int)min((i64)CB, f.sz - (i64)k * CB); };
  // counters of a matrix: rows of L, preparations of a step, D, rows of U
  auto ctl_of = [&](int b) { return f.ctl + FLOW_HEAD_INTS + (i64)b * f.ctl_stride; };
  auto rowL = [&](int b, int i) { return ctl_of(b) + i; };
  auto prep = [&](int b, int k) { return ctl_of(b) + T + k; };
  auto doneD = [&](int b) { return ctl_of(b) + 2 * T; };
  auto xmaxbits = [&](int b) { return ctl_of(b) + 2 * T + 1; };
  auto rowU = [&](int b, int I) { return ctl_of(b) + 2 * T + 2 + I; };
  // entries of the square of matrix b's Gram matrix as the product left it: this thread's 16 of tile (i, k) (zeros
  // beyond the square) ...
  auto raw_tile = [&](int b, int i, int k, float (&v)[4][4]) {
    const int nr = cols_of(i) - tl.row, nc = cols_of(k) - tl.col;
    const i64 e = (f.o + (i64)i * CB + tl.row) * ld + f.o + (i64)k * CB + tl.col;
    const float* p = (f.part == nullptr ? f.A : f.part) + (i64)b * f.wstride + e;
    const int n = f.part == nullptr ? 1 : f.nsplit;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int x = 0; x < 4; ++x) v[j][x] = 0.f;
    // (four partial sums' loads in flight: one after another, 16 partial sums of the first three tiles were 19 us of latency)
#pragma unroll 1
    for (int q = 0; q < n; q += 4, p += 4 * ld * ld) {
      float w[4][4][4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int dr = 8 * h, dc = 16 * j;
            const float* e = p + u * ld * ld + dr * ld + dc;
            if (VEC) {      // (cols is even; whole sectors: with single words the CTA moved twice the bytes)
              const float2 t = (q + u < n && dr < nr && dc < nc) ? __ldcg(reinterpret_cast<const float2*>(e)) : make_float2(0.f, 0.f);
              w[u][j][2 * h] = t.x; w[u][j][2 * h + 1] = t.y;
            } else {
              w[u][j][2 * h] = (q + u < n && dr < nr && dc < nc) ? __ldcg(e) : 0.f;
              w[u][j][2 * h + 1] = (q + u < n && dr < nr && dc + 1 < nc) ? __ldcg(e + 1) : 0.f;
            }
          }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int x = 0; x < 4; ++x) v[j][x] += w[u][j][x];
    }
    if (f.part != nullptr && f.alpha_dev != nullptr) {
      const float al = f.alpha_dev[(i64)b * f.alpha_stride];
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int x = 0; x < 4; ++x) v[j][x] *= al;
    }
  };
  // ... and of a rows x cols block at p (leading dimension ld), from L2: other CTAs have written it
  auto get_tile = [&](const float* p, int rows, int cols, float (&v)[4][4]) {
    p += (i64)tl.row * ld + tl.col;
    const int nr = rows - tl.row, nc = cols - tl.col;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int dr = 8 * h, dc = 16 * j;
        if (VEC) {
          const float2 t = (dr < nr && dc < nc) ? __ldcg(reinterpret_cast<const float2*>(p + dr * ld + dc)) : make_float2(0.f, 0.f);
          v[j][2 * h] = t.x; v[j][2 * h + 1] = t.y;
        } else {
          v[j][2 * h] = (dr < nr && dc < nc) ? __ldcg(p + dr * ld + dc) : 0.f;
          v[j][2 * h + 1] = (dr < nr && dc + 1 < nc) ? __ldcg(p + dr * ld + dc + 1) : 0.f;
        }
      }
  };
  auto store_tile = [&](float* p, int rows, int cols, const float (&v)[4][4]) {
    p += (i64)tl.row * ld + tl.col;
    const int nr = rows - tl.row, nc = cols - tl.col;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int dr = 8 * h, dc = 16 * j;
        if (VEC) {      // (cols is even)
          if (dr < nr && dc < nc) *reinterpret_cast<float2*>(p + dr * ld + dc) = make_float2(v[j][2 * h], v[j][2 * h + 1]);
        } else {
          if (dr < nr && dc < nc) p[dr * ld + dc] = v[j][2 * h];
          if (dr < nr && dc + 1 < nc) p[dr * ld + dc + 1] = v[j][2 * h + 1];
        }
      }
  };
  auto wait_all = [&](const int* p, int want) -> bool {      // every thread: thread 0 waits, all learn the outcome
    if (tid == 0) s_ok = flow_wait(p, want, f);
    bar_named<1, FLOW_COMPUTE>();
    const bool ok = s_ok >= 0;
    bar_named<1, FLOW_COMPUTE>();
    return ok;
  };
  if (tid == 0) s_ok = 0;
  __syncthreads();

  bool alive = true;
  if ((int)blockIdx.x < f.nb) {
    // ------------------------------------------------------------------------------------------ runner of matrix b
    // The compute threads (eight warps) step from block to block; the service warps beside them wait for the helpers'
    // preparations, bring the next step's operands into shared memory and publish what is finished, so that no
    // wait, load or fence is left on the chain but the barriers between the two.
    const int b = (int)blockIdx.x;
    int* os = f.os + (i64)b * OS_SLOT_INTS;
    if (!skipped(b)) {
      float* G = f.L + (i64)b * f.wstride;
      float* gdiag = f.gdiag + (i64)b * f.wstride;
      float* Dinv = f.Dinv + (i64)b * f.wstride;
      float* DinvP = f.DinvP + (i64)b * f.wstride;
      ctile_t TS[2] = {SA[0], SA[1]};                     // A'_{k,k-1}, then L_{k,k-1}; by parity of k
      ctile_t Lb = SB[0], X = SB[1], C = SC[0];              // the diagonal block; D; A'_kk
      auto tile_at = [&](int i, int k) { return G + (f.o + (i64)i * CB) * ld + f.o + (i64)k * CB; };
      const int lane = tid & 31;
      // reference values of block k's pivots: diag(A) as the product left it
      auto setup = [&](int k, float g0, float g1) {      // (one warp)
        const float inf = __int_as_float(0x7f800000);
        const bool bad = !(fabsf(g0) < inf) || !(fabsf(g1) < inf);
        if (__any_sync(0xffffffffu, bad) && lane == 0 && reinterpret_cast<volatile int*>(os)[OS_FAIL] == 0) {   // (a known failure is not reported twice)
          os[OS_FAIL] = 1;
          atomicOr(f.status_always, DION_STATUS_NONFINITE);
        }
        potrf64_setup(s_set[k & 1], g0, g1, f.floor_rel, lane);
      };
      auto diag_of = [&](int k, int e) { return (e < cols_of(k)) ? __ldcg(gdiag + f.o + (i64)k * CB + e) : 0.f; };
      if (tid >= FLOW_COMPUTE) {
        // ---------------------------------------------------------------- service warps: the first one decides
        const int sid = tid - FLOW_COMPUTE, swarp = sid >> 5;
        if (sid == 0) {
          if (f.o == 0) { os[OS_FLOORED] = 0; os[OS_MINREL] = 0x7f800000; }      // (+inf)
          if (f.exclusive) {
            const unsigned sm = flow_smid();
            atomicOr(f.ctl + FLOW_SM_BITS + (sm >> 5), 1 << (sm & 31));
          }
        }
        bar_named<5, FLOW_THREADS>();      // the first blocks' diagonals are in s_diag
        if (swarp == 0) setup(0, s_diag[0][lane], s_diag[0][lane + 32]);
        if (swarp == 1 && T > 1) setup(1, s_diag[1][lane], s_diag[1][lane + 32]);
        for (int k = 0; k <= T; ++k) {
          bar_named<6, FLOW_THREADS>();      // step k may start: its operands are there; D_{k-1} is stored
          if (s_ok < 0) break;
          if (k > 0 && sid == 0) flow_publish(doneD(b), k);
          if (k == T) break;
          if (k > 0) {
            bar_named<7, FLOW_THREADS>();      // L_{k,k-1} is stored
            if (sid == FLOW_SERVICE - 1) flow_publish(rowL(b, k), k);      // (row k of L is complete)
          }
          if (k + 1 < T && k + 1 >= 2) {
            if (sid == 0) s_prep = flow_wait(prep(b, k + 1), 2, f);
            bar_named<8, FLOW_SERVICE>();
            if (s_prep < 0) {
              if (sid == 0) s_ok = -1;
            } else {
              const int nk = cols_of(k + 1);
              flow_load<VEC, FLOW_SERVICE>(TS[(k + 1) & 1], tile_at(k + 1, k), ld, nk, CB, sid);
              flow_load<VEC, FLOW_SERVICE>(C, tile_at(k + 1, k + 1), ld, nk, nk, sid);
              flow_commit();
              if (swarp == 0) setup(k + 1, diag_of(k + 1, lane), diag_of(k + 1, lane + 32));
              flow_wait_all();
            }
          }
        }
      } else {
        // ---------------------------------------------------------------- compute threads
        float c[4][4];
        {
          float v1[4][4], c1[4][4];
          raw_tile(b, 0, 0, c);
          if (T > 1) { raw_tile(b, 1, 0, v1); raw_tile(b, 1, 1, c1); }
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int x = 0; x < 4; ++x)
              if (tl.r(x) == tl.c(j, x)) {
                s_diag[0][tl.r(x)] = f.gdiag_given ? diag_of(0, tl.r(x)) : c[j][x];
                if (T > 1) s_diag[1][tl.r(x)] = f.gdiag_given ? diag_of(1, tl.r(x)) : c1[j][x];
              }
          if (T > 1) { tile_put(TS[1], tl, v1); tile_put(C, tl, c1); }
        }
        bar_named<5, FLOW_THREADS>();
        for (int k = 0; k <= T; ++k) {
          bar_named<6, FLOW_THREADS>();
          if (s_ok < 0) { alive = false; break; }
          if (k == T) break;
          const int nk = cols_of(k);
          if (k > 0) {
            // L_{k,k-1} = A' D_{k-1}^T (the deflated rows of D zeroed), then the last term of the diagonal block
            tile_get(C, tl, c);
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {      // (one copy of the product's code)
              float v[4][4];
              tile_nt(TS[k & 1], h == 0 ? X : TS[k & 1], h == 0 ? MM_TRI : MM_LOWER, tid, v);
              if (h == 0) {
                bar_named<1, FLOW_COMPUTE>();
                tile_put(TS[k & 1], tl, v);
                store_tile(tile_at(k, k - 1), nk, CB, v);
                bar_named<7, FLOW_THREADS>();
              } else {
#pragma unroll
                for (int j = 0; j < 4; ++j)
#pragma unroll
                  for (int x = 0; x < 4; ++x) c[j][x] -= v[j][x];
              }
            }
          }
          const Potrf64Set& set = s_set[k & 1];
          const float s2 = set.s2;
#pragma unroll
          for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int x = 0; x < 4; ++x) c[j][x] = (tl.r(x) == tl.c(j, x) && tl.r(x) >= nk) ? 1.f : c[j][x] * s2;      // (identity padding)
          tile_put(Lb, tl, c);
          bar_named<1, FLOW_COMPUTE>();
          const i64 d = (i64)(f.o / CB + k) * (CB * CB);
          potrf64(Lb, X, set, aux, f.floor_rel, os, f.status, tid, Dinv + d, DinvP + d);
        }
      }
    }
    __syncthreads();
    alive = s_ok >= 0;
    __syncthreads();
  }
  // -------------------------------------------------------------------------------------------------- helper tasks
  // thread 0 walks the task list: single-matrix positions, every position once per matrix of the chain
  int step = 0;
  int base = 0;      // position of the first task of `step`
  // tasks of list step s: the preparations for the runner's steps up to s + 2 + ahead, the factor's tiles of step s, the
  // panel's of step s - LAG
  auto step_tasks = [&](int s, int& nS, int& nL, int& nP) {
    nL = max(T - 3 - s, 0);
    nS = (s == 0) ? 2 * min(max(T - 2, 0), f.ahead + 1) : 2 * min(max(T - 2 - s - f.ahead, 0), 1);
    nP = 0;
    const int k = s - FLOW_LAG;
    if (k >= 0 && k < T) nP = solve ? NR : flow_inverse_rows(T, k, f.sz < f.r);
  };
  auto fetch_task = [&](int ticket) -> FlowTask {
    FlowTask t;
    t.b = ticket % f.nb;
    const int pos = ticket / f.nb;
    t.type = FT_NONE; t.i = t.k = 0;
    while (step < T + FLOW_LAG) {
      int nS, nL, nP;
      step_tasks(step, nS, nL, nP);
      if (pos < base + nS + nL + nP) {
        int e = pos - base;
        if (e < nS) {
          t.type = (e & 1) ? FT_DIAG : FT_SUB;
          t.i = t.k = (step == 0) ? 2 + (e >> 1) : step + 2 + f.ahead;
        } else if ((e -= nS) < nL) {
          t.type = FT_L; t.i = step + 3 + e; t.k = step;
        } else {
          t.type = FT_PANEL; t.k = step - FLOW_LAG;
          t.i = e - nL;
        }
        return t;
      }
      base += nS + nL + nP;
      ++step;
    }
    return t;
  };
  const int* sm_bits = (f.exclusive && (int)blockIdx.x >= f.nb) ? f.ctl + FLOW_SM_BITS + (flow_smid() >> 5) : nullptr;
  while (alive && tid < FLOW_COMPUTE) {
    if (tid == 0) {
      FlowTask none;
      none.type = FT_NONE; none.b = none.i = none.k = 0;
      s_task = (sm_bits != nullptr && ((flow_ld(sm_bits) >> (flow_smid() & 31)) & 1)) ? none : fetch_task(atomicAdd(f.ctl + FLOW_TICKET, 1));
    }
    bar_named<1, FLOW_COMPUTE>();
    const FlowTask t = s_task;
    if (t.type == FT_NONE) break;
    const int b = t.b;
    if (skipped(b)) { bar_named<1, FLOW_COMPUTE>(); continue; }
    float* G = f.L + (i64)b * f.wstride + f.o * ld + f.o;
    const float* Dk = ((t.type == FT_PANEL) ? f.Dinv : f.DinvP) + (i64)b * f.wstride + (i64)(f.o / CB + ((t.type == FT_SUB || t.type == FT_DIAG) ? t.k - 2 : t.k)) * (CB * CB);
    float* U = f.Pout + (i64)b * f.wstride + (solve ? f.o : f.o * ld + f.o);
    // The tile (i, kt): rows of L or of U, row kt of L they meet, terms j0 .. kt - 1, then D_kt; a preparation goes on to
    // the tile (i, kw): the same terms with row kw, then term kt itself.
    const bool panel = t.type == FT_PANEL, prepares = t.type == FT_SUB || t.type == FT_DIAG, same = t.type == FT_DIAG;
    const int kt = prepares ? t.k - 2 : t.k;
    const int kw = same ? t.k : t.k - 1;
    const int j0 = (panel && !solve) ? t.i : 0;
    const int nrow = (panel && solve) ? (int)min((i64)CB, f.rows - (i64)t.i * CB) : cols_of(t.i);
    const int ncol = cols_of(kt);
    const float* Abase = panel ? U + (i64)t.i * CB * ld : G + (i64)t.i * CB * ld;
    const float* Bbase = G + (i64)kt * CB * ld;
    const float* Wbase = G + (i64)kw * CB * ld;      // (SUB; a whole row block)
    const int* fa = panel ? rowU(b, t.i) : rowL(b, t.i);
    const int* fb = rowL(b, kt);
    const int* fw = rowL(b, kw);
    if (panel && !solve && t.i > t.k) {      // below the block diagonal of L^-T: zeros (the products read whole tiles)
      const float z[4][4] = {};
      store_tile(U + (i64)t.i * CB * ld + (i64)t.k * CB, nrow, ncol, z);
      bar_named<1, FLOW_COMPUTE>();
      continue;
    }
    float v[4][4], w[4][4];      // the tiles' own entries, less the terms
    if (panel && solve) {
      get_tile(f.Pin + (i64)b * f.wstride + (i64)t.i * CB * ld + f.o + (i64)t.k * CB, nrow, ncol, v);
    } else if (panel) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int x = 0; x < 4; ++x) v[j][x] = (t.i == t.k && tl.r(x) == tl.c(j, x)) ? 1.f : 0.f;
    } else {
      raw_tile(b, t.i, kt, v);
    }
    if (prepares) {
      raw_tile(b, t.i, kw, w);
      if (same && !f.gdiag_given) {      // for the pivot floors of the runner
        float* gdiag = f.gdiag + (i64)b * f.wstride + f.o + (i64)t.k * CB;
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
          for (int x = 0; x < 4; ++x)
            if (tl.r(x) == tl.c(j, x) && tl.r(x) < nrow) gdiag[tl.r(x)] = w[j][x];
      }
    }
    int pa = 0, pb = 0, pw = 0;      // progress of the rows as thread 0 has seen it
    const bool other = t.type == FT_SUB;      // a third row of tiles
    auto issue = [&](int j, int st) {
      flow_load<VEC>(SA[st], Abase + (i64)j * CB, ld, nrow, CB, tid);
      flow_load<VEC>(SB[st], Bbase + (i64)j * CB, ld, ncol, CB, tid);
      if (other) flow_load<VEC>(SC[st], Wbase + (i64)j * CB, ld, CB, CB, tid);
      flow_commit();
    };
    auto have = [&](int j) -> bool {      // (thread 0) the tiles of term j are there, as far as can be seen now
      if (pa <= j) pa = flow_ld(fa);
      if (pb <= j) pb = flow_ld(fb);
      if (other && pw <= j) pw = flow_ld(fw);
      return min(pa, pb) > j && (!other || pw > j);
    };
    auto need = [&](int j) -> bool {      // every thread: wait for term j
      if (tid == 0) {
        int ok = 0;
        if (pa <= j) { pa = flow_wait(fa, j + 1, f); ok = min(ok, pa); }
        if (ok >= 0 && pb <= j) { pb = flow_wait(fb, j + 1, f); ok = min(ok, pb); }
        if (ok >= 0 && other && pw <= j) { pw = flow_wait(fw, j + 1, f); ok = min(ok, pw); }
        s_ok = ok;
      }
      bar_named<1, FLOW_COMPUTE>();
      const bool ok = s_ok >= 0;
      bar_named<1, FLOW_COMPUTE>();
      return ok;
    };
    if (j0 < kt) {
      if (!need(j0)) { alive = false; break; }
      issue(j0, 0);
    }
    int st = 0;
    for (int j = j0; j < kt + (prepares ? 2 : 1); ++j) {      // terms, the product with D, a preparation's last term: one copy of the code
      const bool more = j + 1 < kt;
      if (j < kt) {
        if (tid == 0 && more) s_ready[j & 1] = have(j + 1) ? 1 : 0;
        flow_wait_all();
        bar_named<1, FLOW_COMPUTE>();      // term j has landed; everyone is done with the other stage
      } else {
        if (same && j > kt) store_tile(G + (i64)t.i * CB * ld + (i64)kt * CB, nrow, ncol, v);      // (DIAG: L_{k,k-2})
        bar_named<1, FLOW_COMPUTE>();      // everyone is done with the stages
        if (same && j > kt && tid == FLOW_COMPUTE - 1) flow_publish(rowL(b, t.i), kt + 1);
        st = 0;
        tile_put(SA[0], tl, v);
        if (j == kt) {
          if (!wait_all(doneD(b), kt + 1)) { alive = false; break; }
          flow_load<true>(SB[0], Dk, CB, CB, CB, tid);
        } else if (other) {
          if (!wait_all(fw, kt + 1)) { alive = false; break; }
          flow_load<VEC>(SB[0], Wbase + (i64)kt * CB, ld, CB, CB, tid);
        }
        flow_commit();
        flow_wait_all();
        bar_named<1, FLOW_COMPUTE>();
      }
      const bool rdy = more && s_ready[j & 1] != 0;
      if (rdy) issue(j + 1, st ^ 1);
      const int nprod = (prepares && j < kt) ? 2 : 1;
#pragma unroll 1
      for (int q = 0; q < nprod; ++q) {
        float s[4][4];
        const bool self = same && (q == 1 || j > kt);
        tile_nt(SA[st], self ? SA[st] : q == 0 ? SB[st] : SC[st], j == kt ? MM_TRI : self ? MM_LOWER : MM_FULL, tid, s);
        const bool into_w = q == 1 || j > kt;
#pragma unroll
        for (int y = 0; y < 4; ++y)
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            if (into_w) w[y][x] -= s[y][x];
            else v[y][x] = (j == kt) ? s[y][x] : v[y][x] - s[y][x];
          }
      }
      if (more && !rdy) {
        if (!need(j + 1)) { alive = false; break; }
        issue(j + 1, st ^ 1);
      }
      st ^= 1;
    }
    if (!alive) break;
    if (panel && !solve && f.xmax != nullptr) {      // (a maximum: the order of arrival does not matter)
      float m = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int x = 0; x < 4; ++x) m = fmaxf(m, fabsf(v[q][x]));
      const unsigned u = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
      if ((tid & 31) == 0) atomicMax(xmaxbits(b), (int)u);
    }
    if (prepares) store_tile(G + (i64)t.i * CB * ld + (i64)kw * CB, nrow, cols_of(kw), w);
    else store_tile((panel ? U : G) + (i64)t.i * CB * ld + (i64)t.k * CB, nrow, ncol, v);
    bar_named<1, FLOW_COMPUTE>();
    if (tid == 0) {
      if (t.type == FT_L) flow_publish(rowL(b, t.i), t.k + 1);
      else if (panel) { if (t.k + 1 < T) flow_publish(rowU(b, t.i), t.k + 1); }
      else {
        asm volatile("fence.acq_rel.gpu;" ::: "memory");
        atomicAdd(prep(b, t.k), 1);
      }
    }
  }
  // ------------------------------------------------------------------------------------------------------ the end
  __syncthreads();
  if (tid == 0) {
    asm volatile("fence.acq_rel.gpu;" ::: "memory");
    s_ok = (atomicAdd(f.ctl + FLOW_LEFT, 1) == (int)gridDim.x - 1) ? 1 : 0;
  }
  __syncthreads();
  if (s_ok == 0) return;
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
  const bool aborted = flow_ld(f.ctl + FLOW_ABORT) != 0;
  __syncthreads();
  if (f.xmax != nullptr)
    for (int b = tid; b < f.nb; b += FLOW_THREADS)
      if (!skipped(b)) f.xmax[(i64)b * f.wstride] = __int_as_float(flow_ld(xmaxbits(b)));
  __syncthreads();
  const int nints = FLOW_HEAD_INTS + f.nb * f.ctl_stride;
  for (int e = tid; e < nints; e += FLOW_THREADS) f.ctl[e] = 0;
  for (int b = tid; b < f.nb; b += FLOW_THREADS) {
    int* os = f.os + (i64)b * OS_SLOT_INTS;
    if (skipped(b)) continue;
    if (aborted) { os[OS_FAIL] = 1; continue; }
    if (f.round_end == 0) continue;
    round_evaluate(os, f.good_rel, f.done_rel, f.rounds_total);
  }
}

}  // namespace dion
