// fp32 FMA tiled product with fused operand formation and epilogues.
// Takes any shape, stride and alignment; it is the engine for small or ragged
// problems and for the r x r factor updates, and the reference engine the
// tensor-core kernels are compared with.
#pragma once

#include <type_traits>

#include "dion_common.cuh"

namespace dion {

// The matrices of a chain whose operands lie at no common stride: one launch, blockIdx.z = matrix * splits + split; partial sums
// g.bs2 floats apart.  inner > 1 (splits == 1): the block takes all `inner` splits of K of its tile, one after another, and adds
// their sums as k_splitk_reduce would.
struct GemmTabs { const void *A[GEMM_TAB_MAX], *A2[GEMM_TAB_MAX], *B[GEMM_TAB_MAX], *C[GEMM_TAB_MAX], *C2[GEMM_TAB_MAX]; };
struct NoTabs {};
// Two products of the same shape that write different arrays: blockIdx.z tells them apart (no splits, no batch).
struct GemmSecond { GemmArgs g; };

template <int BM, int BN, int BK, int TM, int TN, int MINB, typename TABS>
__global__ void __launch_bounds__(256, MINB) k_gemm_simt(const __grid_constant__ GemmArgs first, const __grid_constant__ TABS tabs, int inner) {
  pdl_enter();
  constexpr bool TWO = std::is_same<TABS, GemmSecond>::value;
  const GemmArgs* args = &first;
  if constexpr (TWO) { if (blockIdx.z != 0) args = &tabs.g; }
  const GemmArgs& g = *args;
  static_assert((BM / TM) * (BN / TN) == 256, "256 threads per tile");
  static_assert(TM % 4 == 0 && TN % 4 == 0, "micro tile in groups of 4");
  // blockIdx.z = inner batch index + batch * outer batch index (or the K split)
  i64 batch = 0, outer = 0;
  int split = 0;
  constexpr bool TAB = std::is_same<TABS, GemmTabs>::value;
  if (TAB) { outer = blockIdx.z / g.splits; split = blockIdx.z % g.splits; }      // (splits: those of the grid)
  else if (!TWO && g.splits > 1) split = blockIdx.z;
  else if (!TWO) { batch = blockIdx.z % g.batch; outer = blockIdx.z / g.batch; }
  if (g.skip_flag != nullptr && g.skip_flag[outer * g.skip_stride] != 0) return;

  constexpr int LDA_S = BM + 4, LDB_S = BN + 4;
  constexpr int A_PER = BM * BK / 256, B_PER = BN * BK / 256;
  constexpr int GM = TM / 4, GN = TN / 4;          // groups of 4 rows / cols per thread
  constexpr int SM_STRIDE = BM / GM, SN_STRIDE = BN / GN;
  __shared__ __align__(16) float As[BK][LDA_S];
  __shared__ __align__(16) float Bs[BK][LDB_S];
  __shared__ float T[BM / GM][BN + 1];

  const int tid = threadIdx.x;
  const int tx = tid % (BN / TN), ty = tid / (BN / TN);
  const i64 i0 = (i64)blockIdx.y * BM, j0 = (i64)blockIdx.x * BN;
  if (g.tri == TRI_LOWER && j0 > i0 + BM - 1) return;

  i64 k_begin = 0, k_end = g.K;
  i64 per = g.K;      // k of one split
  if (g.klimit) k_end = min(g.K, j0 + BN);
  if (g.splits * inner > 1) {
    per = (g.K + g.splits * inner - 1) / (g.splits * inner);
    per = (per + 15) / 16 * 16;
  }
  if (g.splits > 1) {
    k_begin = min(g.K, per * split);
    k_end = min(k_end, k_begin + per);
  }

  const float *A, *B;
  const void *A2 = g.A2, *C2 = g.C2;
  float* C = nullptr;
  if constexpr (TAB) {
    A = reinterpret_cast<const float*>(tabs.A[outer]); B = reinterpret_cast<const float*>(tabs.B[outer]);
    A2 = tabs.A2[outer]; C2 = tabs.C2[outer];
    C = reinterpret_cast<float*>(const_cast<void*>(tabs.C[outer]));
    if (g.splits > 1) C = g.part + outer * g.bs2 + (i64)split * g.M * g.N;
  } else {
    A = g.A + batch * g.bsA + outer * g.bs2; B = g.B + batch * g.bsB + outer * g.bs2;
    C = g.splits > 1 ? g.part + (i64)split * g.M * g.N : g.C + batch * g.bsC + outer * g.bs2;
  }
  const bool a_kcontig = (g.a_sk == 1);
  const bool b_ncontig = (g.b_sn == 1);

  float acc[TM][TN];
#pragma unroll
  for (int a = 0; a < TM; ++a)
#pragma unroll
    for (int b = 0; b < TN; ++b) acc[a][b] = 0.f;

  float ra[A_PER], ra2[A_PER], rb[B_PER];

  // A thread's elements of a K step: one base address and a constant step between them (rows, or k, 256 / BK or 256 / BM apart).
  // (64-bit index arithmetic per element was half of the instructions of a step.)
  const int a_i = a_kcontig ? tid / BK : tid % BM, a_k = a_kcontig ? tid % BK : tid / BM;
  const int b_j = b_ncontig ? tid % BN : tid / BK, b_k = b_ncontig ? tid / BN : tid % BK;
  const int a_di = a_kcontig ? 256 / BK : 0, a_dk = a_kcontig ? 0 : 256 / BM;
  const int b_dj = b_ncontig ? 0 : 256 / BK, b_dk = b_ncontig ? 256 / BN : 0;
  const i64 a_step = a_di * g.a_si + a_dk * g.a_sk, a2_step = a_di * g.a2_si + a_dk * g.a2_sk, b_step = b_dk * g.b_sk + b_dj * g.b_sn;
  const i64 a2_off = (i0 + a_i) * g.a2_si + (k_begin + a_k) * g.a2_sk;
  const float* pa = A + (i0 + a_i) * g.a_si + (k_begin + a_k) * g.a_sk;
  const float* pb = B + (k_begin + b_k) * g.b_sk + (j0 + b_j) * g.b_sn;
  const int m_left = (int)min((i64)BM, g.M - i0), n_left = (int)min((i64)BN, g.N - j0);
  auto fetch = [&](i64 kb) {
    const int k_left = (int)min((i64)BK, k_end - kb);
    const i64 adv = kb - k_begin;
    const float* qa = pa + adv * g.a_sk;
    const float* qb = pb + adv * g.b_sk;
#pragma unroll
    for (int l = 0; l < A_PER; ++l)
      ra[l] = (a_i + l * a_di < m_left && a_k + l * a_dk < k_left) ? qa[l * a_step] : 0.f;
    if (g.a2_mode == ADD_F32) {
      const float* q2 = reinterpret_cast<const float*>(A2) + a2_off + adv * g.a2_sk;
#pragma unroll
      for (int l = 0; l < A_PER; ++l) ra2[l] = (a_i + l * a_di < m_left && a_k + l * a_dk < k_left) ? q2[l * a2_step] : 0.f;
    } else if (g.a2_mode == ADD_BF16) {
      const __nv_bfloat16* q2 = reinterpret_cast<const __nv_bfloat16*>(A2) + a2_off + adv * g.a2_sk;
#pragma unroll
      for (int l = 0; l < A_PER; ++l)
        ra2[l] = (a_i + l * a_di < m_left && a_k + l * a_dk < k_left) ? __bfloat162float(q2[l * a2_step]) : 0.f;
    }
#pragma unroll
    for (int l = 0; l < B_PER; ++l)
      rb[l] = (b_j + l * b_dj < n_left && b_k + l * b_dk < k_left) ? qb[l * b_step] : 0.f;
  };
  auto stage = [&]() {
#pragma unroll
    for (int l = 0; l < A_PER; ++l) {
      const int idx = tid + l * 256;
      const int ii = a_kcontig ? idx / BK : idx % BM;
      const int kk = a_kcontig ? idx % BK : idx / BM;
      As[kk][ii] = g.a2_mode != ADD_NONE ? ra[l] + ra2[l] : ra[l];
    }
#pragma unroll
    for (int l = 0; l < B_PER; ++l) {
      const int idx = tid + l * 256;
      const int jj = b_ncontig ? idx % BN : idx / BK;
      const int kk = b_ncontig ? idx / BN : idx % BK;
      Bs[kk][jj] = rb[l];
    }
  };

  if (k_begin < k_end) fetch(k_begin);
  constexpr bool INNER = TAB && TM * TN <= 16;
  float tot[INNER ? TM : 1][INNER ? TN : 1];
  i64 next = k_begin + per;      // where the next split begins
  if constexpr (INNER) {
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
      for (int b = 0; b < TN; ++b) tot[a][b] = 0.f;
  }
  for (i64 kb = k_begin; kb < k_end; kb += BK) {
    if constexpr (INNER) {
      if (kb == next) {
        next += per;
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
          for (int b = 0; b < TN; ++b) { tot[a][b] += acc[a][b]; acc[a][b] = 0.f; }
      }
    }
    stage();
    __syncthreads();
    if (kb + BK < k_end) fetch(kb + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[TM], b[TN];
#pragma unroll
      for (int gm = 0; gm < GM; ++gm) {
        const float4 v = *reinterpret_cast<const float4*>(&As[kk][gm * SM_STRIDE + ty * 4]);
        a[gm * 4 + 0] = v.x; a[gm * 4 + 1] = v.y; a[gm * 4 + 2] = v.z; a[gm * 4 + 3] = v.w;
      }
#pragma unroll
      for (int gn = 0; gn < GN; ++gn) {
        const float4 v = *reinterpret_cast<const float4*>(&Bs[kk][gn * SN_STRIDE + tx * 4]);
        b[gn * 4 + 0] = v.x; b[gn * 4 + 1] = v.y; b[gn * 4 + 2] = v.z; b[gn * 4 + 3] = v.w;
      }
#pragma unroll
      for (int x = 0; x < TM; ++x)
#pragma unroll
        for (int y = 0; y < TN; ++y) acc[x][y] = fmaf(a[x], b[y], acc[x][y]);
    }
    __syncthreads();
  }

  if constexpr (INNER) {
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
      for (int b = 0; b < TN; ++b) acc[a][b] += tot[a][b];
  }
  float alpha = g.alpha;
  if (g.alpha_dev != nullptr) alpha *= g.alpha_dev[TAB ? outer * g.alpha_dev_stride : 0];

  // The tile goes through shared memory row by row, so that a warp accesses whole row segments, and the loads of C and of the
  // second operand are all issued before the first store (element by element each store waited for its own load, and the
  // next load for that store: 16 times the latency of memory).
  const i64 ldc = g.splits > 1 ? g.N : g.ldc;
  const int epi = g.splits > 1 ? EPI_STORE : g.epi;
  const float scale = g.splits > 1 ? 1.f : alpha;
  constexpr int SLAB = BM / GM;      // rows of the tile per pass (those of one register group of every thread)
  constexpr int PER = SLAB * BN / 256;
  constexpr int RSTEP = 256 / BN;
  const int tc = tid % BN, tr = tid / BN;
#pragma unroll
  for (int gm = 0; gm < GM; ++gm) {
    if (gm > 0) __syncthreads();
#pragma unroll
    for (int x = 0; x < 4; ++x)
#pragma unroll
      for (int y = 0; y < TN; ++y) T[ty * 4 + x][(y / 4) * SN_STRIDE + tx * 4 + (y % 4)] = acc[gm * 4 + x][y];
    __syncthreads();
    const i64 gj = j0 + tc;
    if (gj < g.N) {
      constexpr int BATCH = PER < 16 ? PER : 16;
#pragma unroll 1
      for (int q0 = 0; q0 < PER; q0 += BATCH) {
        float c[BATCH], t[BATCH];
        const i64 r0 = i0 + gm * SM_STRIDE + tr + q0 * RSTEP;
        const int left = (int)min((i64)(BATCH * RSTEP), g.M - r0);      // rows q * RSTEP below it exist
        const float* cp = C + r0 * ldc + gj;
        const i64 c2_off = r0 * g.ldc2 + gj;
        const bool with_c = epi == EPI_SUB || epi == EPI_ADD2_SUB;
        if (with_c) {
#pragma unroll
          for (int q = 0; q < BATCH; ++q) c[q] = q * RSTEP < left ? cp[q * RSTEP * ldc] : 0.f;
        }
        if (epi == EPI_C2_SUB || (epi == EPI_ADD2_SUB && g.c2_mode == ADD_F32)) {
          const float* p = reinterpret_cast<const float*>(C2) + c2_off;
#pragma unroll
          for (int q = 0; q < BATCH; ++q) t[q] = q * RSTEP < left ? p[q * RSTEP * g.ldc2] : 0.f;
        } else if (epi == EPI_ADD2_SUB && g.c2_mode == ADD_BF16) {
          const __nv_bfloat16* p = reinterpret_cast<const __nv_bfloat16*>(C2) + c2_off;
#pragma unroll
          for (int q = 0; q < BATCH; ++q) t[q] = q * RSTEP < left ? __bfloat162float(p[q * RSTEP * g.ldc2]) : 0.f;
        } else {
#pragma unroll
          for (int q = 0; q < BATCH; ++q) t[q] = 0.f;
        }
#pragma unroll
        for (int q = 0; q < BATCH; ++q) {
          if (q * RSTEP >= left) break;
          const float v = T[tr + (q0 + q) * RSTEP][tc];      // (an explicit FMA: the same bits from every instance of this kernel)
          C[(r0 + q * RSTEP) * ldc + gj] = epi == EPI_STORE ? scale * v : fmaf(-scale, v, with_c ? c[q] + t[q] : t[q]);
        }
      }
    }
  }
}

// Sums split-K partials in a fixed order: C = alpha * sum_s part[s].
static __global__ void k_splitk_reduce(const float* __restrict__ part, int splits, i64 M, i64 N,
                                float* __restrict__ C, i64 ldc, float alpha, int tri, int tile,
                                const int* skip_flag, i64 bstride, i64 skip_stride,
                                const float* __restrict__ alpha_dev = nullptr, i64 alpha_dev_stride = 0) {
  // blockIdx.y: the matrix of a batched product (partials and output bstride elements apart)
  pdl_enter();
  if (skip_flag != nullptr && skip_flag[(i64)blockIdx.y * skip_stride] != 0) return;
  if (alpha_dev != nullptr) alpha *= alpha_dev[(i64)blockIdx.y * alpha_dev_stride];
  part += (i64)blockIdx.y * bstride;
  C += (i64)blockIdx.y * bstride;
  const i64 total = M * N;
  if (N % 4 == 0 && ldc % 4 == 0 && (((uintptr_t)C | (uintptr_t)part) & 15) == 0) {      // four elements at a time
    const i64 pr = N / 4;
    for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total / 4; e += (i64)gridDim.x * blockDim.x) {
      const i64 i = row_of(e, pr), j = (e - i * pr) * 4;
      if (tri == TRI_LOWER && (j / tile) > (i / tile)) continue;  // tiles that were never computed
      float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
      for (int p = 0; p < splits; ++p) {
        const float4 v = *reinterpret_cast<const float4*>(part + (i64)p * total + 4 * e);
        s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
      }
      *reinterpret_cast<float4*>(C + i * ldc + j) = make_float4(alpha * s.x, alpha * s.y, alpha * s.z, alpha * s.w);
    }
    return;
  }
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    const i64 i = row_of(e, N), j = e - i * N;
    if (tri == TRI_LOWER && (j / tile) > (i / tile)) continue;
    float s = 0.f;
#pragma unroll 8
    for (int p = 0; p < splits; ++p) s += part[(i64)p * total + e];
    C[i * ldc + j] = alpha * s;
  }
}

}  // namespace dion
