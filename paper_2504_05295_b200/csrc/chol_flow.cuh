// The Cholesky factorization of a Gram matrix, the inverse of its factor and the triangular solve of a panel, as ONE
// launch of cooperating CTAs (data flow between 64 x 64 tiles instead of one launch per block column).
#pragma once

#include <stddef.h>

#include "dion_common.cuh"
#include "umma_ptx.cuh"

namespace dion {

// ---------------------------------------------------------------------------------------------------------------
// fp32 products of bf16 ones: x = h + m + l with h, m, l bf16 (8 + 8 + 8 significant bits, every remainder rounded to nearest), six
// of the nine cross products (those dropped are below 2^-26 of the product).  The h h terms go to one accumulator, the rest to
// others that are added at the end: one truncating add per K step on the main sum.  As accurate as a chain of fp32 FMAs.  Inside a
// diagonal block they are on the warp-level path (mma.sync: an operand fragment of a 16 x 8 tile is a few words per lane, and a
// shared-memory load returns at most 128 bytes a cycle to the registers of an SM, broadcast or not, which held a 64^3 product
// with 4 x 4 outputs per thread at 3900 cycles); products of whole tiles are further below.
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

// ---------------------------------------------------------------------------------------------------------------
// Products on the tensor cores: C = A B^T of tiles whose rows are contiguous along k, 64 of them, each as three bf16 planes (h, m, l)
// of 128 bytes a row (128-byte swizzle), with the six cross products above.  A has 128 rows, the lanes of TMEM; where a tile has
// 64, the MMA also reads the 64 rows behind a plane, whatever lies there, and nothing reads the lanes they go to.
// (mma.sync took 3900 cycles for such a product on eight warps, bound by splitting an operand's fragments in every warp that
// reads them; here an operand is split once and the MMAs, 768 cycles of operand reads, run beside the next operands' split.)
// ---------------------------------------------------------------------------------------------------------------
constexpr uint32_t PLANE = 64 * 128, PLANES = 3 * PLANE;      // bytes
__device__ __forceinline__ uint32_t plane_at(int row, int col) {      // byte offset of an entry (its 8-column unit swizzled)
  return (uint32_t)(row * 128 + ((((col >> 3) ^ row) & 7) << 4) + (col & 7) * 2);
}
__device__ __forceinline__ void planes_put4(uint32_t base, int row, int col, float4 x, uint32_t plane = PLANE) {      // col a multiple of 4
  const Bf3 p = split3(x.x, x.y), q = split3(x.z, x.w);
  const uint32_t a = base + plane_at(row, col);
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(p.h), "r"(q.h) : "memory");
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a + plane), "r"(p.m), "r"(q.m) : "memory");
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a + 2 * plane), "r"(p.l), "r"(q.l) : "memory");
}
// (The pieces below that are called from several places are functions of their own: what a launch costs on a small matrix is to a
// good part the fetching of its code.)
// One thread: the product of the planes at a and b into the TMEM columns d .. d + 191.  The planes of b lie behind one another, so
// that one MMA takes an operand of 64, 128 or 192 rows of them: what bounds these small MMAs is reading their operands from shared
// memory (A's 128 rows 32 cycles, 64 rows of B 16), and A's planes are read once each.  Three accumulators: h h; h m + m h;
// h l + m m + l h.
static __device__ __noinline__ void planes_mma(uint32_t d, uint32_t a, uint32_t b, uint32_t plane_a) {
#pragma unroll
  for (uint32_t k = 0; k < 128; k += 32) {      // bytes of 16 columns
    const uint64_t bd = umma::make_desc<true>(b + k, false, 0);
    const uint32_t more = k != 0 ? 1u : 0u;
    umma::umma<true>(d, umma::make_desc<true>(a + k, false, 0), bd, umma::make_idesc(true, false, false, 192), more);
    umma::umma<true>(d + 64, umma::make_desc<true>(a + plane_a + k, false, 0), bd, umma::make_idesc(true, false, false, 128), 1u);
    umma::umma<true>(d + 128, umma::make_desc<true>(a + 2 * plane_a + k, false, 0), bd, umma::make_idesc(true, false, false, 64), 1u);
  }
}
// 16 columns of the three accumulators of this lane's row, the small ones added first
__device__ __forceinline__ void planes_take16(uint32_t d, float (&v)[16]) {
  uint32_t r[48];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%48];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%49];\n\t"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47}, [%50];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
        "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]),
        "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47])
      : "r"(d), "r"(d + 64), "r"(d + 128)
      : "memory");
#pragma unroll
  for (int e = 0; e < 16; ++e) v[e] = (__uint_as_float(r[32 + e]) + __uint_as_float(r[16 + e])) + __uint_as_float(r[e]);
}
// The entries of a product that a thread reads: a row of TMEM is a lane, and a warp
// reaches the 32 lanes of its rank mod 4.  Of eight warps, w and w + 4 hold rows 32 w .. 32 w + 31, the first four columns 0 .. 31.
struct RowLane {
  int row, col;
  uint32_t tm;      // TMEM offset of its columns
  bool owner;       // of a tile of 64 rows
  __device__ __forceinline__ RowLane(int tid)
      : row(32 * ((tid >> 5) & 3) + (tid & 31)), col(32 * ((tid >> 7) & 1)), tm(((uint32_t)(32 * ((tid >> 5) & 3)) << 16) + (uint32_t)col),
        owner((tid >> 5 & 2) == 0) {}
};
// ... of the diagonal block: Lb = s2 (C - the product), identity beyond n rows (whole warps; d == ~0: no product)
static __device__ __noinline__ void planes_diag(uint32_t d, const float* C, float* Lb, float s2, int row, int col, int n) {
#pragma unroll 1
  for (int h = 0; h < 2; ++h, C += 16, Lb += 16, col += 16) {
    float v[16];
    if (d != ~0u) planes_take16(d + 16 * h, v);
    else {
#pragma unroll
      for (int e = 0; e < 16; ++e) v[e] = 0.f;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 c = *reinterpret_cast<const float4*>(C + 4 * q);
      float o[4] = {c.x, c.y, c.z, c.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = (row >= n && row == col + 4 * q + e) ? 1.f : (o[e] - v[4 * q + e]) * s2;
      *reinterpret_cast<float4*>(Lb + 4 * q) = make_float4(o[0], o[1], o[2], o[3]);
    }
  }
}
// 32 entries of a product into a row of a tile, or off it (whole warps)
template <bool OFF>
static __device__ __noinline__ void planes_take(uint32_t d, float* p) {
#pragma unroll 1
  for (int h = 0; h < 2; ++h, d += 16, p += 16) {
    float v[16];
    planes_take16(d, v);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float4 o = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      if (OFF) {
        const float4 c = *reinterpret_cast<const float4*>(p + 4 * q);
        o = make_float4(c.x - o.x, c.y - o.y, c.z - o.z, c.w - o.w);
      }
      *reinterpret_cast<float4*>(p + 4 * q) = o;
    }
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
__device__ __forceinline__ void bar_arrive() { asm volatile("bar.arrive %0, %1;" ::"n"(ID), "n"(N) : "memory"); }      // (without waiting)
template <int ID, int N>
__device__ __forceinline__ void bar_named() { asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(N) : "memory"); }

// ... and whether v holds in any of the threads
template <int ID, int N>
__device__ __forceinline__ bool bar_any(bool v) {
  int any;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.s32 p, %1, 0;\n\tbar.red.or.pred q, %2, %3, p;\n\tselp.s32 %0, 1, 0, q;\n\t}"
      : "=r"(any) : "r"((int)v), "n"(ID), "n"(N) : "memory");
  return any != 0;
}

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
// with the solve's products).  With many tiles the launch is bound by the helpers' products: on mma.sync they took 3900 cycles
// each (a 2048^2 panel of full rank, three rounds: 1402 us; on tcgen05, 128 rows to a task, 1101).  With few it is bound by the chain of
// diagonal blocks, 8.3 to 9.8 us each (r = 1024: 157 us), of which potrf64 4.3 (its barriers, 64 dependent columns), the two products
// and the passing of their operands 3.3.  Here the chain
// D_k -> L_{k+1,k} -> A_{k+1,k+1} -> D_{k+1} stays inside ONE CTA (the "runner" of its matrix: two 64^3 products
// and potrf64 per step), and every other tile is a task of a helper CTA, left-looking:
//   L(i,k)    = (A_ik - sum_{j<k} L_ij L_kj^T) D_k^T                       i >= k + 3  (the runner makes i = k + 1)
//   DIAG(k)   = A_kk - sum_{j<k-1} L_kj L_kj^T     for the runner's step k (it adds the last term); also makes L_{k,k-2}
//   SUB(k)    = A_{k,k-1} - sum_{j<k-1} L_kj L_{k-1,j}^T     for the runner's step k; makes L_{k,k-2} for itself: fetched from
//               DIAG it would come one trip through memory later on the chain's second loop, D_{k-2} -> L_{k,k-2} -> step k
//   PANEL(I,k)= (P_Ik - sum_{j<k} U_Ij L_kj^T) D_k^T       (inverse: P = I, the sum starts at j = I)
// L and PANEL take 128 rows at a time: an MMA reads 128 rows of A anyway, row kt of L and D are read and split once for them, and
// what bounds a term is shared memory (768 cycles of operand reads by its MMAs; their split and the sums hide behind).  They fetch
// their operands into registers a term ahead; the preparations, which have three operands, by cp.async.
// A tile's terms are added as soon as their factors exist, in the order of j whoever runs
// the task: the result does not depend on the schedule.  Progress is published as one counter per row of L and U
// (tiles of a row are finished in the order of k) and one for D; a consumer's thread 0 polls with acquire loads.
// Helper tasks are handed out in the order of steps (the panel's a few steps behind the factor's), so a task only
// ever waits for tasks handed out before it and for the runners, which are resident: the launch is cooperative.  Only the
// preparations are handed out `ahead` steps early; they hold no more than half of the helpers.  Every wait, those for the MMAs too,
// has a cycle limit (then DION_STATUS_TIMEOUT and os[OS_FAIL], and every CTA leaves with its TMEM given back).  Waits on other CTAs are
// one thread's; those for the MMAs are every thread's own and may end differently, so a CTA goes on to a task's end and leaves behind
// a barrier that tells all threads whether one of them has lost a wait.
// The last CTA to leave clears the counters for the next launch and evaluates the round (adaptive rounds).
// ---------------------------------------------------------------------------------------------------------------
enum : int { FLOW_TICKET = 0, FLOW_LEFT = 1, FLOW_ABORT = 2, FLOW_HEAD_INTS = 32 };   // head of the control block
constexpr int FLOW_CTL_INTS = 64 * 1024;      // ints of a context's control block (zero between launches)
constexpr int FLOW_COMPUTE = 256;            // threads that compute ...
constexpr int FLOW_SERVICE = 128;            // ... and the service warps of a runner
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
  int prows;                // tiles of rows that a task of the panel takes, 1 or 2
  int ahead;                // steps by which the preparations are handed out early (they take on every term since the first column)
  int near;                 // a matrix whose OS_GOOD is 2 is left alone too (k_near_identity has formed its factor)
  int round_end;            // evaluate the adaptive round
  float good_rel, done_rel;
  int* rounds_total;
  long long limit;
  int lose_cta, lose;       // test hook: the first `lose` threads of that CTA (< 0: of every helper) say that they lost a wait
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

// Tiles are handled by 256 threads, four float4 each: row tid / 16 + 16 q, columns 4 (tid % 16) ...  VEC: 16-byte aligned rows,
// a multiple of four columns.  Reads go to L2: other CTAs have written the data.
__device__ __forceinline__ void flow_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void flow_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
template <bool VEC>
__device__ __forceinline__ float4 flow_ld4(const float* p, int left) {      // left: columns there are
  if (VEC) return left > 0 ? __ldcg(reinterpret_cast<const float4*>(p)) : make_float4(0.f, 0.f, 0.f, 0.f);
  return make_float4(left > 0 ? __ldcg(p) : 0.f, left > 1 ? __ldcg(p + 1) : 0.f, left > 2 ? __ldcg(p + 2) : 0.f, left > 3 ? __ldcg(p + 3) : 0.f);
}
// scale * the sum of n arrays `stride` apart, rows x cols of it, into a tile (zeros elsewhere).  Four arrays' loads in flight: one after
// another, 16 partial sums of the first three tiles were 19 us of latency; one array by itself without the other three's predicates.
template <bool VEC>
static __device__ __noinline__ void flow_tile_in(ctile_t T, const float* __restrict__ src, i64 stride, int n, float scale, i64 ld, int rows, int cols, int tid) {
  const int i = tid >> 4, c = (tid & 15) * 4;
  const float* p = src + (i64)i * ld + c;
  float4 v[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = flow_ld4<VEC>(p + (i64)(16 * q) * ld, i + 16 * q < rows ? cols - c : 0);
#pragma unroll 1
  for (int k = 1; k < n; k += 3) {
    float4 w[3][4];
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
      for (int q = 0; q < 4; ++q) w[u][q] = flow_ld4<VEC>(p + (k + u) * stride + (i64)(16 * q) * ld, (k + u < n && i + 16 * q < rows) ? cols - c : 0);
#pragma unroll
    for (int u = 0; u < 3; ++u)
#pragma unroll
      for (int q = 0; q < 4; ++q) { v[q].x += w[u][q].x; v[q].y += w[u][q].y; v[q].z += w[u][q].z; v[q].w += w[u][q].w; }
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) st4(&T[i + 16 * q][c], make_float4(scale * v[q].x, scale * v[q].y, scale * v[q].z, scale * v[q].w));
}
// A tile on its way to shared memory: 16-byte units `step` bytes apart per q from `at` on, where the thread that asked finds them
// again itself.  (VEC: cp.async, the caller commits and waits.)
template <bool VEC>
static __device__ __noinline__ void flow_bring(unsigned char* at, int step, const float* __restrict__ src, i64 ld, int rows, int cols, int tid) {
  const int i = tid >> 4, c = (tid & 15) * 4;
  const float* p = src + (i64)i * ld + c;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int left = i + 16 * q < rows ? cols - c : 0;
    const float* g = p + (i64)(16 * q) * ld;
    if (VEC) {
      const uint32_t dst = umma::smem_u32(at) + (uint32_t)(q * step);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(left > 0 ? g : src), "r"(left > 0 ? 16 : 0) : "memory");
    } else {
      *reinterpret_cast<float4*>(at + q * step) = flow_ld4<false>(g, left);
    }
  }
}
// ... and from there into planes
static __device__ __noinline__ void flow_split(uint32_t planes, const unsigned char* at, int step, int tid) {
#pragma unroll
  for (int q = 0; q < 4; ++q) planes_put4(planes, (tid >> 4) + 16 * q, (tid & 15) * 4, *reinterpret_cast<const float4*>(at + q * step));
}
constexpr int FLOW_TILE_STEP = 16 * CLD * (int)sizeof(float), FLOW_RAW_STEP = 4096;
__device__ __forceinline__ unsigned char* tile_at4(ctile_t T, int tid) { return reinterpret_cast<unsigned char*>(&T[tid >> 4][(tid & 15) * 4]); }
// rows x cols of a tile to global memory
template <bool VEC>
static __device__ __noinline__ void flow_store(ctile_t T, float* __restrict__ dst, i64 ld, int rows, int cols, int tid) {
  const int i = tid >> 4, c = (tid & 15) * 4;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (i + 16 * q >= rows || c >= cols) continue;
    const float4 v = ld4(&T[i + 16 * q][c]);
    float* p = dst + (i64)(i + 16 * q) * ld + c;
    if (VEC) {
      st4(p, v);
    } else {
      p[0] = v.x;
      if (c + 1 < cols) p[1] = v.y;
      if (c + 2 < cols) p[2] = v.z;
      if (c + 3 < cols) p[3] = v.w;
    }
  }
}

// Shared memory, from a 1024-byte boundary: two stages of operand planes (128 and 64 rows, or, of a preparation, three tiles in the
// first one and tiles on their way in the second's place) and 128 rows of results; a runner has the planes of its three operands and its
// tiles there.
constexpr int FLOW_TILE = CB * CLD * (int)sizeof(float);
constexpr uint32_t FLOW_STAGE = 3 * PLANES;
constexpr uint32_t FLOW_COMING = FLOW_STAGE;
constexpr uint32_t FLOW_RAW = CB * CB * sizeof(float);
constexpr uint32_t FLOW_RESULTS = 2 * FLOW_STAGE;
static_assert(FLOW_COMING + 4 * FLOW_RAW <= FLOW_RESULTS && FLOW_STAGE + 4 * FLOW_TILE <= FLOW_RESULTS, "tiles lie behind the first planes");
constexpr int FLOW_SMEM = 1024 + (int)FLOW_RESULTS + 2 * FLOW_TILE;
constexpr int FLOW_ROWS = 2;                  // tiles of rows that a task of the factor takes, and most of a task of the panel
constexpr int FLOW_TMEM = 512;                // columns: two buffers of a product, or one of a preparation's two
constexpr int FLOW_MMA_THREAD = 64;           // issues the MMAs (of a warp that holds no rows of a 64-row tile)

template <bool VEC>
__global__ void __launch_bounds__(FLOW_THREADS, 1) k_chol_flow(const __grid_constant__ FlowArgs f) {
  pdl_enter();
  auto skipped = [&](int b) -> bool {
    const int* os = f.os + (i64)b * OS_SLOT_INTS;
    return (f.skips && os[OS_DONE] != 0) || (f.near && os[OS_GOOD] == 2);
  };
  if ((f.skips || f.near) && __syncthreads_and((int)threadIdx.x >= f.nb || skipped((int)threadIdx.x))) return;      // (nb <= 64)
  extern __shared__ unsigned char flow_smem[];
  const uint32_t smem0 = (umma::smem_u32(flow_smem) + 1023u) & ~1023u;
  unsigned char* const smem_al = flow_smem + (smem0 - umma::smem_u32(flow_smem));
  auto tile_in = [&](uint32_t off) { return reinterpret_cast<ctile_t>(smem_al + off); };
  const ctile_t V = tile_in(FLOW_RESULTS), Wt = tile_in(FLOW_RESULTS + FLOW_TILE);
  __shared__ uint64_t s_bar[2];      // the products of a TMEM buffer are done
  __shared__ uint32_t s_tmem;
  __shared__ Potrf64Set s_set[2];
  __shared__ Potrf64Aux aux;
  __shared__ int s_ready[2];
  __shared__ int s_ok, s_prep, s_first, s_inv;
  __shared__ FlowTask s_task;
  const int tid = threadIdx.x;
  const RowLane rl(tid);
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
  // tile (i, k) of the square of matrix b's Gram matrix as the product left it
  auto raw_tile = [&](ctile_t W, int b, int i, int k, int t) {
    const bool parts = f.part != nullptr;
    const float* p = (parts ? f.part : f.A) + (i64)b * f.wstride + (f.o + (i64)i * CB) * ld + f.o + (i64)k * CB;
    const float scale = (parts && f.alpha_dev != nullptr) ? f.alpha_dev[(i64)b * f.alpha_stride] : 1.f;
    flow_tile_in<VEC>(W, p, ld * ld, parts ? f.nsplit : 1, scale, ld, cols_of(i), cols_of(k), t);
  };
  auto wait_all = [&](const int* p, int want) -> bool {      // every thread: thread 0 waits, all learn the outcome
    if (tid == 0) s_ok = flow_wait(p, want, f);
    bar_named<1, FLOW_COMPUTE>();
    const bool ok = s_ok >= 0;
    bar_named<1, FLOW_COMPUTE>();
    return ok;
  };
  if (tid == 0) {
    s_ok = s_inv = 0;
    umma::mbar_init(umma::smem_u32(&s_bar[0]), 1);
    umma::mbar_init(umma::smem_u32(&s_bar[1]), 1);
    umma::fence_barrier_init();
  }
  if (tid >= FLOW_COMPUTE && tid < FLOW_COMPUTE + 32) {      // (one service warp; nothing that holds TMEM fits beside this CTA)
    umma::tmem_alloc(umma::smem_u32(&s_tmem), FLOW_TMEM);
    umma::tmem_relinquish();
  }
  umma::tc_fence_before();
  __syncthreads();
  umma::tc_fence_after();
  const uint32_t tmem0 = *reinterpret_cast<volatile uint32_t*>(&s_tmem);
  unsigned phase = 0;      // parities of s_bar, per buffer
  auto tmem_of = [&](int buf) { return tmem0 + (uint32_t)buf * 256u; };
  auto commit = [&](int buf) { umma::umma_commit(umma::smem_u32(&s_bar[buf])); };
  // Every compute thread: the products of `buf` are done, or this thread has lost a wait.
  bool lost = false;
  auto mma_wait = [&](int buf) {
    const uint32_t bar = umma::smem_u32(&s_bar[buf]), par = (phase >> buf) & 1u;
    phase ^= 1u << buf;
    if (!umma::mbar_try_wait(bar, par)) {
      const long long t0 = clock64();
      while (!umma::mbar_try_wait(bar, par))
        if (lost || clock64() - t0 > f.limit) { lost = true; break; }      // (waited for that long once only)
    }
    __syncwarp();      // (the loads from TMEM that follow are a warp's)
    umma::tc_fence_after();
  };
  auto loses = [&]() -> bool { return lost || (tid < f.lose && (f.lose_cta < 0 ? (int)blockIdx.x >= f.nb : (int)blockIdx.x == f.lose_cta)); };
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
      const uint32_t PA = smem0, PX = PA + PLANES, PL = PX + PLANES;      // planes of A'_{k,k-1}, D_{k-1}, L_{k,k-1}
      const ctile_t Lb = tile_in(FLOW_STAGE), X = tile_in(FLOW_STAGE + FLOW_TILE),       // the diagonal block; D
                    TS = tile_in(FLOW_STAGE + 2 * FLOW_TILE);                            // L_{k,k-1}
      auto C = [&](int k) { return (k & 1) != 0 ? V : tile_in(FLOW_STAGE + 3 * FLOW_TILE); };      // A'_kk
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
        }
        auto two = [&](auto go) {      // the work of 256 threads
#pragma unroll 1
          for (int h = 0; h < 2; ++h) go(sid + h * FLOW_SERVICE);
        };
        if (f.part != nullptr && T > 1) two([&](int t) { raw_tile(Wt, b, 1, 0, t); });      // (many loads: beside those of the first block)
        bar_named<5, FLOW_THREADS>();      // the first block is in C
        if (swarp == 0)
          setup(0, f.gdiag_given ? diag_of(0, lane) : C(0)[lane][lane], f.gdiag_given ? diag_of(0, lane + 32) : C(0)[lane + 32][lane + 32]);
        int given = 0;      // (thread 0) inverses that are published
        auto publish_d = [&](int n) {
          if (n > given) { flow_publish(doneD(b), n); given = n; }
        };
        // Waits for a preparation (bit 0: SUB, bit 1: DIAG); an inverse that is finished meanwhile is published at once, not behind
        // the next step's beginning, which may be waiting for the same helpers.
        auto wait_prep = [&](int k, int bit) -> bool {
          if (sid == 0) {
            const long long t0 = clock64();
            s_prep = 0;
            for (unsigned polls = 1; (flow_ld(prep(b, k)) & bit) == 0; ++polls) {
              const int n = *reinterpret_cast<volatile int*>(&s_inv);
              if (n > given) { __threadfence_block(); publish_d(n); }
              if ((polls & 15u) != 0) continue;
              if (flow_ld(f.ctl + FLOW_ABORT) != 0) { s_prep = -1; break; }
              if (clock64() - t0 > f.limit) {
                atomicExch(f.ctl + FLOW_ABORT, 1);
                atomicOr(f.status_always, DION_STATUS_TIMEOUT);
                s_prep = -1;
                break;
              }
            }
          }
          bar_named<8, FLOW_SERVICE>();
          lost = lost || s_prep < 0;      // (every barrier up to the next step's is still met)
          return s_prep >= 0;
        };
        for (int k = 0; k <= T; ++k) {
          // step k may start: A'_{k,k-1} is there, D_{k-1} is stored; and whether it does is the same to every thread
          if (bar_any<6, FLOW_THREADS>(loses())) { alive = false; break; }
          if (sid == 0) publish_d(k);
          if (k == T) break;
          if (k > 0) {
            if (k >= 2 && wait_prep(k, 2)) {      // A'_kk and its pivots' reference values
              const int nk = cols_of(k);
              two([&](int t) { flow_bring<VEC>(tile_at4(C(k), t), FLOW_TILE_STEP, tile_at(k, k), ld, nk, nk, t); });
              flow_commit();
              if (swarp == 0) setup(k, diag_of(k, lane), diag_of(k, lane + 32));
              flow_wait_all();
            }
            bar_arrive<9, FLOW_THREADS>();
            bar_named<7, FLOW_THREADS>();      // L_{k,k-1} is in TS
            two([&](int t) { flow_store<VEC>(TS, tile_at(k, k - 1), ld, cols_of(k), CB, t); });
            bar_named<8, FLOW_SERVICE>();
            if (sid == FLOW_SERVICE - 1) flow_publish(rowL(b, k), k);      // (row k of L is complete)
          }
          if (k + 1 < T) {      // the next step's operand (the products that read A' are over)
            if (k == 0) {
              const ctile_t Cn = C(1);
              two([&](int t) {
                if (f.part == nullptr) raw_tile(Wt, b, 1, 0, t);
                raw_tile(Cn, b, 1, 1, t);
              });
              bar_named<8, FLOW_SERVICE>();
              if (swarp == 0)
                setup(1, f.gdiag_given ? diag_of(1, lane) : Cn[lane][lane], f.gdiag_given ? diag_of(1, lane + 32) : Cn[lane + 32][lane + 32]);
            } else {
              if (!wait_prep(k + 1, 1)) continue;
              two([&](int t) { flow_bring<VEC>(tile_at4(Wt, t), FLOW_TILE_STEP, tile_at(k + 1, k), ld, cols_of(k + 1), CB, t); });
              flow_commit();
              flow_wait_all();
            }
            two([&](int t) { flow_split(PA, tile_at4(Wt, t), FLOW_TILE_STEP, t); });
            umma::fence_proxy_async();
          }
        }
      } else {
        // ---------------------------------------------------------------- compute threads
        raw_tile(C(0), b, 0, 0, tid);
        bar_named<5, FLOW_THREADS>();
        for (int k = 0; k <= T; ++k) {
          if (bar_any<6, FLOW_THREADS>(loses())) { alive = false; break; }
          if (k == T) break;
          const int nk = cols_of(k);
          const Potrf64Set& set = s_set[k & 1];
          if (k > 0) {
            // L_{k,k-1} = A' D_{k-1}^T (the deflated rows of D zeroed), then the last term of the diagonal block
            flow_split(PX, tile_at4(X, tid), FLOW_TILE_STEP, tid);
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
              umma::fence_proxy_async();
              umma::tc_fence_before();
              bar_named<1, FLOW_COMPUTE>();
              if (tid == FLOW_MMA_THREAD) {
                umma::tc_fence_after();
                planes_mma(tmem_of(h), h == 0 ? PA : PL, h == 0 ? PX : PL, PLANE);
                commit(h);
              }
              mma_wait(h);
              if (h == 0) {
                if (rl.owner) planes_take<false>(tmem_of(0) + rl.tm, &TS[rl.row][rl.col]);
                bar_arrive<7, FLOW_THREADS>();      // (the service warps store it)
                bar_named<1, FLOW_COMPUTE>();
                flow_split(PL, tile_at4(TS, tid), FLOW_TILE_STEP, tid);
              }
            }
            bar_named<9, FLOW_THREADS>();      // A'_kk is there
          }
          if (rl.owner) planes_diag(k > 0 ? tmem_of(1) + rl.tm : ~0u, &C(k)[rl.row][rl.col], &Lb[rl.row][rl.col], set.s2, rl.row, rl.col, nk);
          umma::tc_fence_before();
          bar_named<1, FLOW_COMPUTE>();
          const i64 d = (i64)(f.o / CB + k) * (CB * CB);
          potrf64(Lb, X, set, aux, f.floor_rel, os, f.status, tid, Dinv + d, DinvP + d);
          if (tid == 0) { __threadfence_block(); *reinterpret_cast<volatile int*>(&s_inv) = k + 1; }
        }
      }
    }
    __syncthreads();
  }
  // -------------------------------------------------------------------------------------------------- helper tasks
  // thread 0 walks the task list: single-matrix positions, every position once per matrix of the chain
  int step = 0;
  int base = 0;      // position of the first task of `step`
  // tasks of list step s: the preparations for the runner's steps up to s + 2 + ahead, the factor's tiles of step s, the
  // panel's of step s - LAG
  auto step_tasks = [&](int s, int& nS, int& nL, int& nP) {
    nL = (max(T - 3 - s, 0) + FLOW_ROWS - 1) / FLOW_ROWS;
    nS = (s == 0) ? 2 * min(max(T - 2, 0), f.ahead + 1) : 2 * min(max(T - 2 - s - f.ahead, 0), 1);
    nP = 0;
    const int k = s - FLOW_LAG;
    if (k >= 0 && k < T) nP = ((solve ? NR : flow_inverse_rows(T, k, f.sz < f.r)) + f.prows - 1) / f.prows;
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
          t.type = FT_L; t.i = step + 3 + FLOW_ROWS * e; t.k = step;
        } else {
          t.type = FT_PANEL; t.k = step - FLOW_LAG;
          t.i = f.prows * (e - nL);
        }
        return t;
      }
      base += nS + nL + nP;
      ++step;
    }
    return t;
  };
  int ticket = -1;      // (thread 0) drawn at the end of the task before
  while (alive && tid < FLOW_COMPUTE) {
    if (tid == 0) {
      s_task = fetch_task(ticket >= 0 ? ticket : atomicAdd(f.ctl + FLOW_TICKET, 1));
      ticket = -1;
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
    const int nrow = (int)min((i64)(prepares ? CB : (panel ? f.prows : FLOW_ROWS) * CB), (panel && solve ? f.rows : f.sz) - (i64)t.i * CB);
    const int ncol = cols_of(kt);
    const float* Abase = panel ? U + (i64)t.i * CB * ld : G + (i64)t.i * CB * ld;
    const float* Bbase = G + (i64)kt * CB * ld;
    const float* Wbase = G + (i64)kw * CB * ld;      // (SUB; a whole row block)
    const int* fa = panel ? rowU(b, t.i / f.prows) : rowL(b, t.i);
    const int* fb = rowL(b, kt);
    const int* fw = rowL(b, kw);
    if (panel && !solve && t.i > t.k) {      // below the block diagonal of L^-T: zeros (the products read whole tiles)
      float* p = U + (i64)t.i * CB * ld + (i64)t.k * CB;
      for (int e = tid; e < nrow * ncol; e += FLOW_COMPUTE) p[(i64)(e / ncol) * ld + e % ncol] = 0.f;
      bar_named<1, FLOW_COMPUTE>();
      continue;
    }
    // the tiles' own entries (V, Wt: 128 rows, or a preparation's two tiles)
    if (panel) {
      if (solve) {
        const float* src = f.Pin + (i64)b * f.wstride + (i64)t.i * CB * ld + f.o + (i64)t.k * CB;
#pragma unroll 1
        for (int h = 0; h * CB < nrow; ++h) flow_tile_in<VEC>(h == 0 ? V : Wt, src + (i64)h * CB * ld, 0, 1, 1.f, ld, nrow - h * CB, ncol, tid);
      } else {
#pragma unroll
        for (int q = 0; q < 4 * FLOW_ROWS; ++q) {
          const int row = (tid >> 4) + 16 * q, c = (row & (CB - 1)) - (tid & 15) * 4;
          const bool on = t.i + row / CB == t.k;
          st4(&V[row][(tid & 15) * 4], make_float4(on && c == 0 ? 1.f : 0.f, on && c == 1 ? 1.f : 0.f, on && c == 2 ? 1.f : 0.f, on && c == 3 ? 1.f : 0.f));
        }
      }
    } else {
#pragma unroll 1
      for (int h = 0; h < 2; ++h) raw_tile(h == 0 ? V : Wt, b, t.i + (prepares ? 0 : h), prepares && h == 1 ? kw : kt, tid);
    }
    int pa = 0, pb = 0, pw = 0, pd = 0;      // progress of the rows and of D as thread 0 has seen it
    const bool other = t.type == FT_SUB;      // a third row of tiles
    auto have = [&](int j) -> bool {      // (thread 0) the operands of term j are there, as far as can be seen now; term kt: D
      if (j == kt) {
        if (pd <= kt) pd = flow_ld(doneD(b));
        return pd > kt;
      }
      if (pa <= j) pa = flow_ld(fa);
      if (t.type == FT_L && nrow > CB && pa > j) pa = min(pa, flow_ld(fa + 1));
      if (pb <= j) pb = flow_ld(fb);
      if (other && pw <= j) pw = flow_ld(fw);
      return min(pa, pb) > j && (!other || pw > j);
    };
    auto need = [&](int j) -> bool {      // every thread: wait for term j
      if (tid == 0) {
        int ok = 0;
        if (!have(j)) {
          if (j == kt) {
            ok = pd = flow_wait(doneD(b), kt + 1, f);
          } else {
            if (pa <= j) { pa = flow_wait(fa, j + 1, f); ok = min(ok, pa); }
            if (ok >= 0 && t.type == FT_L && nrow > CB) { pa = min(pa, flow_wait(fa + 1, j + 1, f)); ok = min(ok, pa); }
            if (ok >= 0 && pb <= j) { pb = flow_wait(fb, j + 1, f); ok = min(ok, pb); }
            if (ok >= 0 && other && pw <= j) { pw = flow_wait(fw, j + 1, f); ok = min(ok, pw); }
          }
        }
        s_ok = ok;
      }
      bar_named<1, FLOW_COMPUTE>();
      return s_ok >= 0;      // (written again behind a later barrier only)
    };
    auto stage = [&](int buf) { return smem0 + (uint32_t)buf * FLOW_STAGE; };
    if (!prepares) {
      // ---- 128 rows of the factor or of the panel: operands through registers, a term ahead; the rows under way in registers too
      float4 xa[4 * FLOW_ROWS], xb[4];
      const int i0 = tid >> 4, c0 = (tid & 15) * 4;
      auto fetch = [&](int j) {
        const bool d = j == kt;
        if (!d) {
          const float* p = Abase + (i64)i0 * ld + (i64)j * CB + c0;
#pragma unroll
          for (int q = 0; q < 4 * FLOW_ROWS; ++q) xa[q] = flow_ld4<VEC>(p + (i64)(16 * q) * ld, i0 + 16 * q < nrow ? CB : 0);
        }
        const float* p = d ? Dk + i0 * CB + c0 : Bbase + (i64)i0 * ld + (i64)j * CB + c0;
        const i64 lb = d ? CB : ld;
        const int rows = d ? CB : ncol;
#pragma unroll
        for (int q = 0; q < 4; ++q) xb[q] = flow_ld4<VEC>(p + (i64)(16 * q) * lb, i0 + 16 * q < rows ? CB : 0);
      };
      if (tid == 0) s_first = have(j0) ? 1 : 0;
      bar_named<1, FLOW_COMPUTE>();
      bool fetched = s_first != 0;
      if (fetched) fetch(j0);
      float v[32];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const float4 x = ld4(&V[rl.row][rl.col + 4 * q]);
        v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
      }
      auto less = [&](int buf) {      // the products of a term come off
        mma_wait(buf);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float t16[16];
          planes_take16(tmem_of(buf) + rl.tm + 16 * h, t16);
#pragma unroll
          for (int e = 0; e < 16; ++e) v[16 * h + e] -= t16[e];
        }
      };
      int buf = 0;
#pragma unroll 1
      for (int j = j0; j <= kt; ++j) {      // term j's operands are split while the products of term j - 1 run
        if (j == kt) {      // the rows themselves, the last term's product taken off (all before D is waited for)
          if (j > j0) less(buf ^ 1);
#pragma unroll
          for (int q = 0; q < 8; ++q) planes_put4(stage(buf), rl.row, rl.col + 4 * q, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]), 2 * PLANE);
          if (tid == 0) ticket = atomicAdd(f.ctl + FLOW_TICKET, 1);      // (the next one, so that it is there in time)
        }
        if (!fetched) {
          if (!need(j)) {
            if (j > j0 && j < kt) mma_wait(buf ^ 1);      // (the products in flight)
            alive = false;
            break;
          }
          fetch(j);
        }
        if (j < kt) {
#pragma unroll
          for (int q = 0; q < 4 * FLOW_ROWS; ++q) {
            if (q >= 4 && nrow <= CB) break;      // (one tile: the other lanes' products go nowhere)
            planes_put4(stage(buf), i0 + 16 * q, c0, xa[q], 2 * PLANE);
          }
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) planes_put4(stage(buf) + 6 * PLANE, i0 + 16 * q, c0, xb[q]);
        if (tid == 0 && j < kt) s_ready[j & 1] = have(j + 1) ? 1 : 0;
        umma::fence_proxy_async();
        umma::tc_fence_before();
        bar_named<1, FLOW_COMPUTE>();
        if (tid == FLOW_MMA_THREAD) {
          umma::tc_fence_after();
          planes_mma(tmem_of(buf), stage(buf), stage(buf) + 6 * PLANE, 2 * PLANE);
          commit(buf);
        }
        fetched = j < kt && s_ready[j & 1] != 0;
        if (fetched) fetch(j + 1);
        if (j < kt) {
          if (j > j0) less(buf ^ 1);
          buf ^= 1;
        }
      }
      if (!alive) break;
      mma_wait(buf);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float t16[16];
        planes_take16(tmem_of(buf) + rl.tm + 16 * h, t16);
#pragma unroll
        for (int q = 0; q < 4; ++q) st4(&V[rl.row][rl.col + 16 * h + 4 * q], make_float4(t16[4 * q], t16[4 * q + 1], t16[4 * q + 2], t16[4 * q + 3]));
      }
      umma::tc_fence_before();
      if (bar_any<1, FLOW_COMPUTE>(loses())) { alive = false; break; }
      if (panel && !solve && f.xmax != nullptr) {      // (a maximum: the order of arrival does not matter)
        float m = 0.f;
#pragma unroll
        for (int q = 0; q < 4 * FLOW_ROWS; ++q) {
          if (q >= 4 && nrow <= CB) break;
          const float4 x = ld4(&V[i0 + 16 * q][c0]);
          m = fmaxf(m, fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))));
        }
        const unsigned u = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
        if ((tid & 31) == 0) atomicMax(xmaxbits(b), (int)u);
      }
      float* dst = (panel ? U : G) + (i64)t.i * CB * ld + (i64)t.k * CB;
#pragma unroll 1
      for (int h = 0; h * CB < nrow; ++h) flow_store<VEC>(h == 0 ? V : Wt, dst + (i64)h * CB * ld, ld, nrow - h * CB, ncol, tid);
      bar_named<1, FLOW_COMPUTE>();
      if (tid == 0) {
        if (t.type == FT_L) {
          flow_publish(rowL(b, t.i), t.k + 1);
          if (nrow > CB) flow_publish(rowL(b, t.i + 1), t.k + 1);
        } else if (t.k + 1 < T) {
          flow_publish(rowU(b, t.i / f.prows), t.k + 1);
        }
      }
      continue;
    }
    // ---- a preparation
    // Terms j0 .. kt - 1, then, as "term" kt, the product with D.  A term's operands are brought up to two terms ahead.
    // (SUB, one term ahead, keeps its third tile where another's second term would be)
    auto coming = [&](int j) { return smem_al + FLOW_COMING + (other ? 0 : (j - j0) & 1) * 2 * FLOW_RAW + tid * 16; };
    unsigned char* const third = smem_al + FLOW_COMING + 2 * FLOW_RAW + tid * 16;
    auto fetch = [&](int j) {
      unsigned char* at = coming(j);
      if (j < kt) {
        flow_bring<VEC>(at, FLOW_RAW_STEP, Abase + (i64)j * CB, ld, nrow, CB, tid);
        flow_bring<VEC>(at + FLOW_RAW, FLOW_RAW_STEP, Bbase + (i64)j * CB, ld, ncol, CB, tid);
        if (other) flow_bring<VEC>(third, FLOW_RAW_STEP, Wbase + (i64)j * CB, ld, CB, CB, tid);
      } else {
        flow_bring<true>(at + FLOW_RAW, FLOW_RAW_STEP, Dk, CB, CB, CB, tid);
      }
      flow_commit();
    };
    // The operands are in the planes: the products of a term, with a tile of row kt and one of row kw, into a TMEM buffer each.
    auto products = [&](bool second) {
      umma::fence_proxy_async();
      umma::tc_fence_before();
      bar_named<1, FLOW_COMPUTE>();
      if (tid == FLOW_MMA_THREAD) {
        umma::tc_fence_after();
        planes_mma(tmem_of(0), stage(0), stage(0) + PLANES, PLANE);
        if (second) planes_mma(tmem_of(1), stage(0), stage(0) + (same ? 0u : 2 * PLANES), PLANE);
        commit(0);
      }
    };
    if (tid == 0) s_first = have(j0) ? (!other && j0 < kt && have(j0 + 1) ? 2 : 1) : 0;
    bar_named<1, FLOW_COMPUTE>();
    if (same && !f.gdiag_given && tid < nrow)      // for the pivot floors of the runner
      f.gdiag[(i64)b * f.wstride + f.o + (i64)t.k * CB + tid] = Wt[tid][tid];
    int fetched = j0 - 1 + s_first;      // the last term whose operands are on their way
    if (fetched >= j0) fetch(j0);
    if (fetched > j0) fetch(j0 + 1);
    float* const vrow = &V[rl.row][rl.col];
    float* const wrow = &Wt[rl.row][rl.col];
#pragma unroll 1
    for (int j = j0; j <= kt; ++j) {
      if (j == kt) {      // the tile itself, every term taken off
        if (j > j0) bar_named<1, FLOW_COMPUTE>();
        flow_split(stage(0), tile_at4(V, tid), FLOW_TILE_STEP, tid);
      }
      if (fetched < j) {
        if (!need(j)) { alive = false; break; }
        fetch(j);
        fetched = j;
      }
      if (fetched > j) asm volatile("cp.async.wait_group 1;" ::: "memory");
      else flow_wait_all();
      unsigned char* at = coming(j);
      if (j < kt) flow_split(stage(0), at, FLOW_RAW_STEP, tid);
      flow_split(stage(0) + PLANES, at + FLOW_RAW, FLOW_RAW_STEP, tid);
      if (other && j < kt) flow_split(stage(0) + 2 * PLANES, third, FLOW_RAW_STEP, tid);
      const int next = fetched + 1;
      const bool ask = next <= kt && next <= j + (other ? 1 : 2);
      if (tid == 0 && ask) s_ready[j & 1] = have(next) ? 1 : 0;
      products(j < kt);
      if (ask && s_ready[j & 1] != 0) { fetch(next); fetched = next; }
      if (j < kt) {      // they come off
        mma_wait(0);
        if (rl.owner) {
          planes_take<true>(tmem_of(0) + rl.tm, vrow);
          planes_take<true>(tmem_of(1) + rl.tm, wrow);
        }
        umma::tc_fence_before();
      }
    }
    if (!alive) break;
    bool w_there = false;      // (SUB: the last term's other operand, made by the runner about now)
    if (other) {
      if (tid == 0) s_first = flow_ld(fw) > kt ? 1 : 0;
      bar_named<1, FLOW_COMPUTE>();
      w_there = s_first != 0;
      if (w_there) { flow_bring<VEC>(third, FLOW_RAW_STEP, Wbase + (i64)kt * CB, ld, CB, CB, tid); flow_commit(); }
    }
    mma_wait(0);
    if (rl.owner) planes_take<false>(tmem_of(0) + rl.tm, vrow);
    umma::tc_fence_before();
    bar_named<1, FLOW_COMPUTE>();
    // ... whose result is the last term's operand (DIAG: and L_{k,k-2})
    flow_split(stage(0), tile_at4(V, tid), FLOW_TILE_STEP, tid);
    if (other) {
      if (!w_there) {
        if (!wait_all(fw, kt + 1)) { alive = false; break; }
        flow_bring<VEC>(third, FLOW_RAW_STEP, Wbase + (i64)kt * CB, ld, CB, CB, tid);
        flow_commit();
      }
      flow_wait_all();
      flow_split(stage(0) + PLANES, third, FLOW_RAW_STEP, tid);
    }
    umma::fence_proxy_async();
    bar_named<1, FLOW_COMPUTE>();
    if (tid == FLOW_MMA_THREAD) {
      umma::tc_fence_after();
      planes_mma(tmem_of(1), stage(0), stage(0) + (other ? PLANES : 0u), PLANE);
      commit(1);
    }
    if (same) {
      flow_store<VEC>(V, G + (i64)t.i * CB * ld + (i64)kt * CB, ld, nrow, ncol, tid);
      bar_named<1, FLOW_COMPUTE>();
      if (tid == FLOW_COMPUTE - 1) flow_publish(rowL(b, t.i), kt + 1);
    }
    mma_wait(1);
    if (rl.owner) planes_take<true>(tmem_of(1) + rl.tm, wrow);
    umma::tc_fence_before();
    if (bar_any<1, FLOW_COMPUTE>(loses())) { alive = false; break; }
    flow_store<VEC>(Wt, G + (i64)t.i * CB * ld + (i64)kw * CB, ld, nrow, cols_of(kw), tid);
    bar_named<1, FLOW_COMPUTE>();
    if (tid == 0) {
      asm volatile("fence.acq_rel.gpu;" ::: "memory");
      atomicAdd(prep(b, t.k), same ? 2 : 1);
    }
  }
  if (!alive && loses()) {
    atomicExch(f.ctl + FLOW_ABORT, 1);
    atomicOr(f.status_always, DION_STATUS_TIMEOUT);
  }
  // ------------------------------------------------------------------------------------------------------ the end
  umma::tc_fence_before();
  __syncthreads();
  if (tid >= FLOW_COMPUTE && tid < FLOW_COMPUTE + 32) {
    umma::tc_fence_after();
    umma::tmem_dealloc(tmem0, FLOW_TMEM);
  }
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
