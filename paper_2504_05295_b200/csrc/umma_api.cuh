// Host interface of the tensor-core engine (umma_gemm.cuh, compiled in a unit of its own: its kernels take minutes).
#pragma once

#include "dion_common.cuh"

namespace dion {
namespace umma {
constexpr long long SPIN_LIMIT_CYCLES = 2000000000LL;  // cycle budget of a bounded wait: about one second
// CTA pairs that can be resident at once on the current device (0: no pairs).
int pair_clusters(int sm_count);
}  // namespace umma

// One-time set-up of the tensor-core kernels: opt in to their dynamic shared memory.
int umma_configure();

// Shapes the tensor engine may take (alignment decides the rest).
inline bool umma_shape_ok(const GemmArgs& g, int precision) {
  const int epc = (g.ab16 || precision == DION_PREC_BF16_OPERANDS) ? 8 : 4;
  return g.M >= 128 && g.N >= 64 && g.K >= 64 && g.M % epc == 0 && g.N % epc == 0 && g.K % epc == 0;
}


// Launches the product on the tensor cores if it qualifies.  Returns the number of
// kernels launched (1, or 2 with a split-K reduction), 0 if this engine does not take
// the product, or a negative DION_ERR_* code.
// `variant` (test hook, 0 in the product): UMMA_VARIANT_* bits.
enum : int {
  UMMA_VARIANT_REGISTER_LOADS = 1,   // operands through registers instead of TMA
  UMMA_VARIANT_WITHHOLD = 2,         // with register loads: withhold one producer arrival, 1 ms wait budget
  UMMA_VARIANT_NO_PAIRS = 4,         // single-CTA tiles where the product would take CTA pairs
  UMMA_VARIANT_NO_TMA_EPI = 8        // register epilogue where the product would take the TMA epilogue
};

// K splits of a plain-store product of few tiles: enough for every worker (CTA, or pair of CTAs) to have an item, at least four
// K blocks each.
constexpr i64 UMMA_MAX_SPLITS = 32;
inline i64 umma_split_count(i64 tiles, i64 workers, i64 nkb) {
  i64 want = workers / tiles;
  if (want > nkb / 4) want = nkb / 4;
  return want > UMMA_MAX_SPLITS ? UMMA_MAX_SPLITS : want < 1 ? 1 : want;
}
constexpr i64 UMMA_PAIR_MIN_ROWS = 512;   // smallest output height given to CTA pairs
constexpr i64 UMMA_PAIR_MIN_TRI = 2048;   // smallest lower-triangular output given to CTA pairs
// Floats of partial sums that the splits of an M x N product take in the tiles that its shape usually gets and whole K blocks of 32.  Not
// a bound: a product that its operands keep from CTA pairs (a bf16 addend, no tensor maps) has other tiles and may want more
// splits (600 x 256: 29 against 24), K blocks that are not whole one more; the launch takes as many as the scratch holds.
inline i64 umma_split_floats(i64 M, i64 N, i64 K, bool tri, int sm_count) {
  if (M < 128 || N < 64) return 0;
  const bool pairs = N >= 256 && M >= UMMA_PAIR_MIN_ROWS && (!tri || N >= UMMA_PAIR_MIN_TRI);
  const i64 tm = pairs ? 256 : 128, tn = (N < 256 || (tri && !pairs)) ? 128 : 256;
  const i64 nM = (M + tm - 1) / tm, nN = (N + tn - 1) / tn, tiles = tri ? nM * (nM + 1) / 2 : nM * nN;
  const i64 splits = umma_split_count(tiles, pairs ? sm_count / 2 : sm_count, K / 32);
  return splits > 1 ? splits * M * N : 0;
}
int umma_try_launch(const GemmArgs& g_in, int precision, int sm_count, float* part, i64 part_floats, int* status,
                    cudaStream_t st, int variant = 0);

}  // namespace dion
