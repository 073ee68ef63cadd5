#include "sparq_gemm_small_kernel.cuh"

namespace sparq { SPARQ_DEFINE_GEMM_SMALL(128) }
