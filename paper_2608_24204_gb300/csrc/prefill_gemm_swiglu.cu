// The prefill GEMM kernels with the PEpiSwiGLU epilogue.
#include "prefill_gemm.cuh"

namespace wici {
WICI_GEMM_INSTANCE(, PEpiSwiGLU)
}  // namespace wici
