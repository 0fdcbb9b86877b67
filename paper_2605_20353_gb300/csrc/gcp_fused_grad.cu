// gcp_fused_grad.cu -- the fused kernel's gradient instantiations
// (gcp_fused.cuh), in their own translation unit so that they compile beside
// the others.
#include "gcp_fused.cuh"

namespace gcpk {

int fused_max_blocks(int d, bool bf16, int cols) {
    switch (d) {
    case 2: return fused_occupancy_d<2, false>(bf16, cols);
    case 3: return fused_occupancy_d<3, false>(bf16, cols);
    case 4: return fused_occupancy_d<4, false>(bf16, cols);
    case 5: return fused_occupancy_d<5, false>(bf16, cols);
    case 6: return fused_occupancy_d<6, false>(bf16, cols);
    case 7: return fused_occupancy_d<7, false>(bf16, cols);
    case 8: return fused_occupancy_d<8, false>(bf16, cols);
    default: return num_sms();
    }
}

// Samples per warp tile: with r = ceil(S / (32 W)) rounds of tiles over the W
// resident warps, the smallest tile that still takes r rounds (a multiple of
// the samples that the warp's groups evaluate at once), so that every warp
// has the same work: 250,000 samples on 4,864 warps are two rounds of 28
// instead of one of 32 and 0.6 of another, and small sets spread over all
// warps.
int fused_tile(int64_t S, int log2L, int max_blocks) {
    const int64_t warps = (int64_t)max_blocks * kWarps;
    const int ngrp = 32 >> log2L;
    const int64_t rounds = (S + 32 * warps - 1) / (32 * warps);
    if (rounds < 1) return 32;
    const int64_t per = (S + warps * rounds - 1) / (warps * rounds);
    return (int)((per + ngrp - 1) / ngrp * ngrp);
}

cudaError_t launch_fused(const FusedSpec &f, bool bf16, int cols, int max_blocks, cudaStream_t st,
                         int *blocks_used) {
    return launch_fused_any<false>(f, bf16, cols, max_blocks, st, blocks_used);
}

}  // namespace gcpk
