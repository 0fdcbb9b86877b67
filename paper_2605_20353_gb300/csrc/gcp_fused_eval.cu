// gcp_fused_eval.cu -- the fused kernel's instantiations without reductions
// (gcp_fused.cuh): the loss alone, or the gradient tensor written out for a
// separate MTTKRP.
#include "gcp_fused.cuh"

namespace gcpk {

cudaError_t launch_fused_eval(const FusedSpec &f, bool bf16, int cols, int max_blocks, cudaStream_t st,
                              int *blocks_used) {
    return launch_fused_any<true>(f, bf16, cols, max_blocks, st, blocks_used);
}

}  // namespace gcpk
