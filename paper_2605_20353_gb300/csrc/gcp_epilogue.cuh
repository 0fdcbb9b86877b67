// gcp_epilogue.cuh -- the hot-row replica fold shared by the step epilogues
// (k_post_step for one context, k_batch_post for a batch of clients).
//
// The fused pass sends the gradient reductions of rows that many samples hit
// to NREP replicas of each; the epilogue adds them into the row's gradient
// before Adam.  A hot quad (four columns of a hot row) has
// NREP replica quads; loaded one after another they cost a memory round trip
// per group, so instead a group of NREP / 4 lanes takes one hot quad, four
// replicas a lane, and every replica load is in flight at once.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gcpe {

template <int NREP>
__host__ __device__ constexpr int hot_lanes() {  // lanes that fold one hot quad together
    return NREP / 4;
}

// Sum of the NREP replica quads at R4, R4 + step, R4 + 2 step, ... over a
// group of H = NREP / 4 lanes: lane l of the group loads replicas l, l + H,
// l + 2 H, l + 3 H, adds them in that order, then the group sums its lanes
// with a butterfly (offsets H/2, ..., 1).  The order is fixed, so the result
// does not vary from run to run.  Every lane returns the total; each lane
// clears the replicas it loaded.  All lanes of the group must call it
// together (gmask = the group's lanes).
template <int NREP>
__device__ __forceinline__ float4 hot_quad_sum(float4 *__restrict__ R4, int step, unsigned gmask) {
    constexpr int H = hot_lanes<NREP>();
    static_assert(4 * H == NREP && H <= 32, "four replicas a lane");
    const int l = threadIdx.x & (H - 1);
    float4 v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = R4[(l + H * i) * step];
    float4 t = v[0];
#pragma unroll
    for (int i = 1; i < 4; ++i) {
        t.x += v[i].x;
        t.y += v[i].y;
        t.z += v[i].z;
        t.w += v[i].w;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) R4[(l + H * i) * step] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
    for (int off = H / 2; off > 0; off >>= 1) {
        t.x += __shfl_xor_sync(gmask, t.x, off);
        t.y += __shfl_xor_sync(gmask, t.y, off);
        t.z += __shfl_xor_sync(gmask, t.z, off);
        t.w += __shfl_xor_sync(gmask, t.w, off);
    }
    return t;
}

// Mask of the lane group of the calling lane.
template <int NREP>
__device__ __forceinline__ unsigned hot_group_mask() {
    constexpr int H = hot_lanes<NREP>();
    return (unsigned)((1ull << H) - 1ull) << ((threadIdx.x & 31) & ~(H - 1));
}

}  // namespace gcpe
