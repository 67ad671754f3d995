// The tensor-core engine's kernels and their launches.
#include <string.h>

#include "umma_gemm.cuh"
