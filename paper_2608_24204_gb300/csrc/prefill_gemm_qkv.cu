// The prefill GEMM kernels with the PEpiQKV epilogue.
#include "prefill_gemm.cuh"

namespace wici {
WICI_GEMM_INSTANCE(, PEpiQKV)
}  // namespace wici
