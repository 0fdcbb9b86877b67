// gcp_fused.cuh -- the fused stochastic GCP gradient on sm_103a.
//
// One pass per sample set (the fused Sampling-MTTKRP of Sec. 3.1.2, here with
// stratified sampling and hash rejection):
//   phase A, one sample per lane: Philox4x64-10 counters -> nonzero record
//            load, or zero candidates probed against the nonzero hash set
//            until one is absent (Sec. 3.1.1);
//   phase B, one sample per group of L = Rp / COLS lanes: each lane gathers
//            16-byte slices of the d factor rows, forms the CP model
//            entry m (Eq. cp) with a shuffle reduction over the group,
//            evaluates f and f', and scatters w f' prod_{k!=n} A_k(i_k,:)
//            into every mode's gradient row with FP32 vector reductions
//            (Eq. gcp-gradient, atomic MTTKRP of Sec. 3.1.2).
// The sampled loss is accumulated in FP64 per lane, reduced per block into
// a partials array and finished by a single block in fixed order.
// Gradient passes and passes without reductions (the loss alone, or the
// gradient tensor written out) are separate instantiations, compiled in
// their own translation units (gcp_fused_grad.cu, gcp_fused_eval.cu).
#pragma once

#include <cuda_bf16.h>

#include "gcp_device.cuh"
#include "gcp_internal.h"

namespace gcpk {

using namespace gcpdev;

constexpr int kThreads = 256;

inline int num_sms() {
    static int sms = 0;
    if (!sms) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    }
    return sms;
}

template <int D>
__device__ __forceinline__ void draw_tuple(const SampleSpec &S, uint64_t stream, uint64_t j, uint64_t sub0,
                                           int32_t (&idx)[D]) {
#pragma unroll
    for (int b = 0; 4 * b < D; ++b) {
        const U64x4 w = philox4x64_10(j, sub0 + (uint64_t)b, S.iter, 0, S.seed, stream);
#pragma unroll
        for (int k = 4 * b; k < D && k < 4 * b + 4; ++k)
            idx[k] = (int32_t)map_range32(w.v[k - 4 * b], (uint32_t)S.dims[k]);
    }
}

template <int D>
__device__ __forceinline__ uint64_t linear_of(const SampleSpec &S, const int32_t (&idx)[D]) {
    uint64_t L = 0;
#pragma unroll
    for (int k = 0; k < D; ++k) L += (uint64_t)(uint32_t)idx[k] * S.stride[k];
    return L;
}

template <int D>
__device__ __forceinline__ void load_record(const int32_t *__restrict__ rec, uint64_t e, int32_t (&idx)[D],
                                            float &x) {
    constexpr int NV = (D + 4) / 4;  // 16-byte vectors holding D coordinates + value
    constexpr int RW = rec_words_for(D);
    const int4 *r = reinterpret_cast<const int4 *>(rec + e * RW);
    int w[4 * NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
        const int4 t = __ldg(r + v);
        w[4 * v] = t.x;
        w[4 * v + 1] = t.y;
        w[4 * v + 2] = t.z;
        w[4 * v + 3] = t.w;
    }
#pragma unroll
    for (int k = 0; k < D; ++k) idx[k] = w[k];
    x = __int_as_float(w[D]);
}

// ------------------------------------------------------------ fused pass
// Per warp and per tile of P.tile <= 32 consecutive samples (fused_tile):
//   A1 (tile t+1, one sample per lane): Philox draw; the nonzero record, the
//      dense value or the first hash bucket of the zero candidate is copied
//      into shared memory with cp.async while tile t is processed;
//   A2 (tile t): finish the draw -- a zero candidate found in its bucket is
//      rejected and redrawn with direct probes (rare: 1/(1-N/M) attempts);
//   B  (tile t, one sample per group of L = Rp/COLS lanes): lane g owns
//      COLS columns as COLS/4 quads (4g..4g+3, and Rp/2+4g.. when COLS = 8),
//      so a group's loads and vector reductions cover whole 32-byte sectors
//      and, for rows up to 128 bytes, one whole row per instruction.  Quads
//      beyond the rank hold zeros and are not reduced; they are loaded, as
//      a test around the loads costs more than the sectors (orders 2 to 8,
//      ranks 20 to 65, 2^20 samples: 0 to 15% slower with it).
// The loss: the group's first lane leaves f in shared memory, in words that
// nothing else uses during phase B (the stage's hash buckets, all read by
// then: the other lanes of the group may still be reading the sample's slot);
// after the tile each lane takes its own sample's f.  Without reductions
// (EVAL) no lane of the group needs f', so the group leaves m there and each lane
// evaluates its own sample: one evaluation per tile instead of one per group
// round, and the gradient tensor's entries written by neighbouring lanes
// (2^19 samples of the 4-way Zipf counts in BF16, a loss call: 48.1 -> 45.3
// us; deterministic gradient of 2^21 samples at rank 64: 531 -> 501 us, 494
// with the losses added as follows).
// Each lane adds its sample's f to its own FP64 totals (nonzero and other
// samples apart), one FP64 addition per tile and warp.  They are slow here,
// 16 cycles of the SM's pipe for a warp, so the lanes' totals meet at the end
// in few instructions (block_totals): with five shuffle steps for each of the
// two totals in every warp a pass of 10,000 samples took 2 us more than with
// FP32 sums of each tile, with block_totals 0.3 us more (8.6 -> 8.9 us per
// iteration of a fit), and passes of 2^18 samples and more take less, as a tile
// no longer has five shuffle steps (dense 5-way gradient of 2^22 samples 329 ->
// 324 us).  A sample's m is summed per quad, then
// over quads Rp / 2 columns apart, then Rp / 4, ..., whatever COLS is, and a
// sample's lane and warp depend on the tile alone, so a loss pass and a
// gradient pass over the same samples give the same loss bit for bit
// although they split rows differently.
// Gradient rows that many samples hit go to one of the call's nrep replicas
// (chosen by warp), folded into G afterwards, so that the reductions of hot
// rows do not serialise on one address; with nrep = 0 (few samples) every
// row is added to G itself.
constexpr int kWarps = kThreads / 32;

// The block's sums of its threads' a and b and of the warps' counts n, in a
// fixed order, to out[0..2] (n is the same in every lane of a warp).  Lanes 0
// to 15 of a warp take its a, lanes 16 to 31 its b, one addition for both; then
// one warp adds the warps' rows in pairs and the halves of the result: 19
// additions of a warp a block, in chains of 8.  scratch: kWarps rows of 33
// doubles, free for use by the whole block.
__device__ __forceinline__ void block_totals(double a, double b, int n, double (*scratch)[33], double *out) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool low = lane < 16;
    const double other = __shfl_xor_sync(0xFFFFFFFFu, low ? b : a, 16);
    scratch[warp][lane] = (low ? a : b) + other;
    if (lane == 0) scratch[warp][32] = __longlong_as_double((long long)n);
    __syncthreads();
    if (warp != 0) return;
    double t[kWarps];
#pragma unroll
    for (int w = 0; w < kWarps; ++w) t[w] = scratch[w][lane];
#pragma unroll
    for (int h = kWarps / 2; h > 0; h >>= 1)
#pragma unroll
        for (int w = 0; w < h; ++w) t[w] += t[w + h];
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) t[0] += __shfl_xor_sync(0xFFFFFFFFu, t[0], o);
    if ((lane & 15) == 0) out[lane >> 4] = t[0];
    if (lane == 1) {
        long long c = 0;
#pragma unroll
        for (int w = 0; w < kWarps; ++w) c += __double_as_longlong(scratch[w][32]);
        out[2] = (double)c;
    }
}

// EVAL: no reductions (P.G null); P.Yval, if set, receives the gradient tensor.
template <int D, typename TF, int COLS, bool EVAL>
__global__ void __launch_bounds__(kThreads, fused_min_blocks(D, EVAL ? 4 : COLS)) k_fused(const FusedSpec P) {
    constexpr int SW = rec_words_for(D);  // words per staged sample: coordinates, value, replica slots
    constexpr int NQ = COLS / 4;          // quads of columns per lane
    __shared__ __align__(16) int32_t s_slot[2][kWarps][32][SW];
    __shared__ __align__(16) uint64_t s_bkt[2][kWarps][32][4];

    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    const int log2L = P.log2L;
    const int L = 1 << log2L;
    const int glane = lane & (L - 1);
    const int grp = lane >> log2L;
    const int ngrp = 32 >> log2L;
    const unsigned gmask = (L == 32) ? 0xFFFFFFFFu : (((1u << L) - 1u) << (grp * L));
    int col[NQ];
    [[maybe_unused]] bool on[NQ];  // the quad holds columns of the rank, not padding alone
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        col[q] = q * (P.Rp >> 1) + 4 * glane;
        on[q] = col[q] < P.R;
    }
    const int p = (int)P.s.p;  // sample counts of one call are below 2^31
    const int S = (int)(P.s.p + P.s.q);
    const unsigned TS = P.tile;
    const int ntiles = (int)(((int64_t)S + TS - 1) / TS);  // S may be 2^31 - 1
    const int nwarps = (gridDim.x * blockDim.x) >> 5;
    const int warp0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const TF *F = static_cast<const TF *>(P.F);
    const bool semi = P.s.sampling == GCP_SAMPLING_SEMI_STRATIFIED;
    const bool uniform = P.s.sampling == GCP_SAMPLING_UNIFORM;
    [[maybe_unused]] float *const grep = P.Grep ? P.Grep + (size_t)(warp0 & (P.nrep - 1)) * P.rplane : nullptr;

    double acc_nz = 0.0, acc_z = 0.0;
    int attempts = 0;

    // A1: start the draw of this lane's sample of `tile` into stage `st`;
    // returns the key of a stratified zero candidate (kEmpty otherwise).
    auto issue = [&](int tile, int st) -> uint64_t {
        if (tile >= ntiles || lane >= (int)TS) return kEmpty;
        const unsigned us = (unsigned)tile * TS + lane;  // may pass 2^31 - 1 in the last tile
        int32_t *slot = s_slot[st][warp][lane];
        if (us >= (unsigned)S) return kEmpty;
        const int s = (int)us;
        if (uniform) {
            int32_t idx[D];
            draw_tuple<D>(P.s, kStreamUniform, (uint64_t)(uint32_t)s, 0, idx);
#pragma unroll
            for (int k = 0; k < D; ++k) slot[k] = idx[k];
            cp_async4(slot + D, P.s.dense + linear_of<D>(P.s, idx));
            return kEmpty;
        }
        if (s < p) {
            const U64x4 w = philox4x64_10((uint64_t)(uint32_t)s, 0, P.s.iter, 0, P.s.seed, kStreamNonzero);
            const int32_t *rec = P.s.rec + map_range(w.v[0], (uint64_t)P.s.nnz) * SW;
#pragma unroll
            for (int v = 0; v < SW / 4; ++v) cp_async16(slot + 4 * v, rec + 4 * v);
            return kEmpty;
        }
        int32_t idx[D];
        draw_tuple<D>(P.s, semi ? kStreamSemiZero : kStreamZero, (uint64_t)(uint32_t)(s - p), 0, idx);
#pragma unroll
        for (int k = 0; k < D; ++k) slot[k] = idx[k];
        slot[D] = 0;  // x = 0.0f
        if (semi) return kEmpty;
        const uint64_t key = linear_of<D>(P.s, idx);
        const uint64_t *b = P.s.hkeys + 4 * (mix64(key) & P.s.hbmask);
        cp_async16(&s_bkt[st][warp][lane][0], b);
        cp_async16(&s_bkt[st][warp][lane][2], b + 2);
        return key;
    };

    // A2: finish the draw of stage `st`; returns whether the sample exists.
    auto finish = [&](int tile, int st, uint64_t key) -> bool {
        const unsigned us = (unsigned)tile * TS + lane;
        if (lane >= (int)TS || us >= (unsigned)S) return false;
        const int s = (int)us;
        if (key == kEmpty) return true;  // nonzero, semi-stratified or dense draw
        const ulonglong2 lo = *reinterpret_cast<const ulonglong2 *>(&s_bkt[st][warp][lane][0]);
        const ulonglong2 hi = *reinterpret_cast<const ulonglong2 *>(&s_bkt[st][warp][lane][2]);
        int h = bucket_decide(lo, hi, key);
        if (h == 2)
            h = hash_contains_from(P.s.hkeys, P.s.hbmask, key, ((mix64(key) & P.s.hbmask) + 1) & P.s.hbmask, 1);
        if (h == 0) {
            attempts += 1;
            return true;
        }
        // rejected: redraw until a candidate is absent (Sec. 3.1.1)
        int32_t *slot = s_slot[st][warp][lane];
        const uint64_t j = (uint64_t)(uint32_t)(s - p);
        for (int a = 1; h == 1 && a < P.s.max_attempts; ++a) {
            int32_t idx[D];
            draw_tuple<D>(P.s, kStreamZero, j, 4 * (uint64_t)a, idx);
            h = hash_contains(P.s.hkeys, P.s.hbmask, linear_of<D>(P.s, idx));
            if (h == 0) {
#pragma unroll
                for (int k = 0; k < D; ++k) slot[k] = idx[k];
                attempts += a + 1;
                return true;
            }
        }
        if (h < 0) {
            atomicOr(P.s.status, kErrHashFull);
        } else {
            attempts += P.s.max_attempts;
            atomicOr(P.s.status, kErrExhausted);
        }
        return false;
    };

    // loss and derivative of one sample
    auto sample_loss = [&](float x, float m, bool is_nz, float &f, float &df) {
        float f1, d1;
        loss_eval(P.loss, x, m, f1, d1);
        if (semi && is_nz) {
            float f0, d0;
            loss_eval(P.loss, 0.0f, m, f0, d0);
            f1 -= f0;
            d1 -= d0;
        }
        f = f1;
        df = d1;
    };

    int tile = warp0;
    uint64_t key_next = issue(tile, 0);
    cp_async_commit();
    // the draws need only what never changes; everything else (factors, G,
    // replicas, the incoming scale, the partials) waits for the grids before.
    // Dependents are let in only then, so that theirs wait for ours alone.
    grid_wait();
    grid_trigger();
    const float scale = P.dscale ? *P.dscale : 1.0f;
    for (int st = 0; tile < ntiles; tile += nwarps, st ^= 1) {
        const uint64_t key = key_next;
        __syncwarp();  // stage st^1 is free: the previous tile's phase B is done
        key_next = issue(tile + nwarps, st ^ 1);
        cp_async_commit();
        cp_async_wait<1>();  // this lane's copies into stage st have landed
        const bool ok = finish(tile, st, key);
        const unsigned okmask = __ballot_sync(0xFFFFFFFFu, ok);
        __syncwarp();  // every lane's staged sample is visible to the warp, and every bucket has been read
        float *const handoff = reinterpret_cast<float *>(&s_bkt[st][warp][0][0]);  // [32]: f (EVAL: m) per sample

        // phase B: one sample per group
        for (int it = 0; it * ngrp < (int)TS; ++it) {
            const int src = it * ngrp + grp;
            if (!((okmask >> src) & 1u)) continue;  // uniform within the group
            const int32_t *slot = s_slot[st][warp][src];
            int32_t ii[D];
#pragma unroll
            for (int k = 0; k < D; ++k) ii[k] = slot[k];

            int off[D];
            float a[D][COLS];
#pragma unroll
            for (int k = 0; k < D; ++k) {
                off[k] = (P.rowoff[k] + ii[k]) * P.Rp;
#pragma unroll
                for (int q = 0; q < NQ; ++q) load_quad_coherent(F + off[k] + col[q], a[k] + 4 * q);
            }
            float suf[D][COLS];  // suf[k] = prod_{j>k} a_j
#pragma unroll
            for (int v = 0; v < COLS; ++v) suf[D - 1][v] = 1.0f;
#pragma unroll
            for (int k = D - 2; k >= 0; --k)
#pragma unroll
                for (int v = 0; v < COLS; ++v) suf[k][v] = suf[k + 1][v] * a[k + 1][v];
            float mq[NQ];  // per quad
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                mq[q] = 0.0f;
#pragma unroll
                for (int v = 4 * q; v < 4 * q + 4; ++v) mq[q] = fmaf(a[0][v], suf[0][v], mq[q]);
            }
            float m = NQ == 2 ? mq[0] + mq[NQ - 1] : mq[0];
            for (int o = L >> 1; o > 0; o >>= 1) m += __shfl_xor_sync(gmask, m, o);

            if constexpr (EVAL) {  // the sample's own lane takes it from here
                if (glane == 0) handoff[src] = m;
            } else {
                const float xs = __int_as_float(slot[D]);
                const bool is_nz = !uniform && ((unsigned)tile * TS + src) < (unsigned)p;
                float f, df;
                sample_loss(xs, m, is_nz, f, df);
                if (glane == 0) handoff[src] = f;
                const float y = ((is_nz || uniform) ? P.w_nz : P.w_z) * df * scale;
                float pre[COLS];
#pragma unroll
                for (int v = 0; v < COLS; ++v) pre[v] = y;
#pragma unroll
                for (int n = 0; n < D; ++n) {
                    // replica slot: stored in a nonzero's record; for drawn
                    // cells, rows of fully replicated modes only.  Passes
                    // without replicas skip the search up to order 4 (rank
                    // 20, 250,000 samples: 27.7 -> 27.1 us); at order 5 the
                    // branch costs registers (dense 5-way: 325 -> 335 us)
                    float *g;
                    if constexpr (D > 4) {
                        unsigned hs;
                        if (is_nz && grep)
                            hs = ((unsigned)slot[D + 1 + n / 2] >> (16 * (n & 1))) & 0xFFFFu;
                        else
                            hs = P.small_base[n] >= 0 ? (unsigned)(P.small_base[n] + ii[n]) : kNoSlot;
                        // orders above 4 keep the replicas in planes: rstride is Rp
                        g = hs != kNoSlot ? grep + (int)hs * P.Rp : P.G + off[n];
                    } else {
                        g = P.G + off[n];
                        if (grep) {
                            unsigned hs;
                            if (is_nz)
                                hs = ((unsigned)slot[D + 1 + n / 2] >> (16 * (n & 1))) & 0xFFFFu;
                            else
                                hs = P.small_base[n] >= 0 ? (unsigned)(P.small_base[n] + ii[n]) : kNoSlot;
                            if (hs != kNoSlot) g = grep + (int)hs * P.rstride;
                        }
                    }
#pragma unroll
                    for (int q = 0; q < NQ; ++q)
                        if (on[q])
                            red_add_v4(g + col[q], pre[4 * q] * suf[n][4 * q], pre[4 * q + 1] * suf[n][4 * q + 1],
                                   pre[4 * q + 2] * suf[n][4 * q + 2], pre[4 * q + 3] * suf[n][4 * q + 3]);
#pragma unroll
                    for (int v = 0; v < COLS; ++v) pre[v] *= a[n][v];
                }
            }
        }
        __syncwarp();  // the losses (EVAL: the models) are handed over
        float fl = ok ? handoff[lane] : 0.0f;
        const unsigned s0 = (unsigned)tile * TS;
        if constexpr (EVAL) {
            const bool is_nz = !uniform && s0 + lane < (unsigned)p;
            float df = 0.0f;
            if (ok) sample_loss(__int_as_float(s_slot[st][warp][lane][D]), fl, is_nz, fl, df);
            if (P.Yval && lane < (int)TS && s0 + lane < (unsigned)S) {
                // the gradient tensor entry; no sample: a zero at a valid cell
                const int64_t sm = s0 + lane;
#pragma unroll
                for (int k = 0; k < D; ++k) P.Ycoord[sm * P.ystride + k] = s_slot[st][warp][lane][k];
                P.Yval[sm * P.vstride] = ok ? ((is_nz || uniform) ? P.w_nz : P.w_z) * df * scale : 0.0f;
            }
        }
        if (uniform || s0 + lane < (unsigned)p)  // apart in one tile at most
            acc_nz += (double)fl;
        else
            acc_z += (double)fl;
    }
    cp_async_wait<0>();

    // the block's FP64 loss sums and attempt count
    attempts = __reduce_add_sync(0xFFFFFFFFu, attempts);
    __syncthreads();  // staging is free now
    block_totals(acc_nz, acc_z, attempts, reinterpret_cast<double(*)[33]>(&s_bkt[0][0][0][0]),
                 P.partials + 4 * blockIdx.x);
}

// Resident blocks, and the launch, of the (dtype, columns) instantiation.
template <int D, typename TF, int COLS, bool EVAL>
int fused_occupancy() {
    static int nb = -1;
    if (nb < 0) {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fused<D, TF, COLS, EVAL>, kThreads, 0);
        nb = (per_sm < 1 ? 1 : per_sm) * num_sms();
    }
    return nb;
}

template <int D, bool EVAL>
int fused_occupancy_d(bool bf16, int cols) {
    if (bf16)
        return cols == 8 ? fused_occupancy<D, __nv_bfloat16, 8, EVAL>() : fused_occupancy<D, __nv_bfloat16, 4, EVAL>();
    return cols == 8 ? fused_occupancy<D, float, 8, EVAL>() : fused_occupancy<D, float, 4, EVAL>();
}

template <int D, typename TF, int COLS, bool EVAL>
cudaError_t launch_fused_k(const FusedSpec &f, int blocks, cudaStream_t st) {
    if (f.dependent) return launch_dependent(k_fused<D, TF, COLS, EVAL>, blocks, kThreads, 0, st, f);
    k_fused<D, TF, COLS, EVAL><<<blocks, kThreads, 0, st>>>(f);
    return cudaGetLastError();
}

template <int D, bool EVAL>
cudaError_t launch_fused_d(const FusedSpec &f, bool bf16, int cols, int blocks, cudaStream_t st) {
    if (bf16)
        return cols == 8 ? launch_fused_k<D, __nv_bfloat16, 8, EVAL>(f, blocks, st)
                         : launch_fused_k<D, __nv_bfloat16, 4, EVAL>(f, blocks, st);
    return cols == 8 ? launch_fused_k<D, float, 8, EVAL>(f, blocks, st)
                     : launch_fused_k<D, float, 4, EVAL>(f, blocks, st);
}

template <bool EVAL>
cudaError_t launch_fused_any(const FusedSpec &f, bool bf16, int cols, int max_blocks, cudaStream_t st,
                             int *blocks_used) {
    const int64_t S = f.s.p + f.s.q;
    const int64_t ntiles = (S + f.tile - 1) / f.tile;
    int64_t want = (ntiles + kWarps - 1) / kWarps;
    if (want < 1) want = 1;
    const int blocks = (int)(want < max_blocks ? want : max_blocks);
    *blocks_used = blocks;
    switch (f.s.d) {
    case 2: return launch_fused_d<2, EVAL>(f, bf16, cols, blocks, st);
    case 3: return launch_fused_d<3, EVAL>(f, bf16, cols, blocks, st);
    case 4: return launch_fused_d<4, EVAL>(f, bf16, cols, blocks, st);
    case 5: return launch_fused_d<5, EVAL>(f, bf16, cols, blocks, st);
    case 6: return launch_fused_d<6, EVAL>(f, bf16, cols, blocks, st);
    case 7: return launch_fused_d<7, EVAL>(f, bf16, cols, blocks, st);
    case 8: return launch_fused_d<8, EVAL>(f, bf16, cols, blocks, st);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace gcpk
