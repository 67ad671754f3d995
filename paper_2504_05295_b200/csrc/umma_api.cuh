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
int umma_try_launch(const GemmArgs& g_in, int precision, int sm_count, float* part, i64 part_floats, int* status,
                    cudaStream_t st, int variant = 0);

}  // namespace dion
