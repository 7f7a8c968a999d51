// The decode step for widths without an instantiation of their own (bf16): the same
// persistent kernel with each phase's shape picked at run time.  Such widths used to run
// as five launches a layer and the LM head, 77 us a layer at hidden 3072, ffn 8192 (24
// heads of 128), against 41 here and 30 of HBM time.  Eight bodies for each of five phases in one kernel spill
// (1.1 to 1.2 KB a thread); twelve warps with 200 registers each take the spills away and
// are no faster (367 to 373 us a step against 366), so the step keeps nine warps.
#include "decode_step.cuh"

namespace wici {

using Any = GShape<1, 1, false>;   // stands for no shape

MegaLaunch mega_any_launcher(int head_dim) {
    return head_dim == 128 ? launch_mega<128, Any, Any, false, Any, Any, true>
                           : launch_mega<64, Any, Any, false, Any, Any, true>;
}

cudaError_t setup_mega_any() {
    const cudaError_t e = mega_smem<128, Any, Any, false, Any, Any, true>();
    return e != cudaSuccess ? e : mega_smem<64, Any, Any, false, Any, Any, true>();
}

}  // namespace wici
