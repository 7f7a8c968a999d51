// The prefill GEMM kernels with the PEpiResidual epilogue.
#include "prefill_gemm.cuh"

namespace wici {
WICI_GEMM_INSTANCE(, PEpiResidual)
}  // namespace wici
