// gcp_kernels.cu -- the kernels around the fused pass (gcp_fused.cuh): the
// sample writer, the epilogues of a gradient call and of a training step,
// Adam, nonzero records, and the non-fused MTTKRP.
#include <cuda_bf16.h>

#include "gcp_device.cuh"
#include "gcp_epilogue.cuh"
#include "gcp_fused.cuh"
#include "gcp_internal.h"

using namespace gcpdev;

namespace gcpk {

static int elementwise_blocks(int64_t n);

struct RowOffsets {
    int64_t off[GCP_MAX_NDIM];
};

// Draw sample s of the set.  Returns false when the sample does not exist
// (exhausted zero draw); idx then holds the last candidate.
template <int D>
__device__ __forceinline__ bool draw_sample(const SampleSpec &S, int64_t s, int32_t (&idx)[D], float &x,
                                            int &attempts) {
    if (S.sampling == GCP_SAMPLING_UNIFORM) {
        draw_tuple<D>(S, kStreamUniform, (uint64_t)s, 0, idx);
        x = __ldg(S.dense + linear_of<D>(S, idx));
        return true;
    }
    if (s < S.p) {
        const U64x4 w = philox4x64_10((uint64_t)s, 0, S.iter, 0, S.seed, kStreamNonzero);
        load_record<D>(S.rec, map_range(w.v[0], (uint64_t)S.nnz), idx, x);
        return true;
    }
    const uint64_t j = (uint64_t)(s - S.p);
    x = 0.0f;
    if (S.sampling == GCP_SAMPLING_SEMI_STRATIFIED) {
        draw_tuple<D>(S, kStreamSemiZero, j, 0, idx);
        return true;
    }
    for (int a = 0; a < S.max_attempts; ++a) {
        draw_tuple<D>(S, kStreamZero, j, 4 * (uint64_t)a, idx);
        const int h = hash_contains(S.hkeys, S.hbmask, linear_of<D>(S, idx));
        if (h == 0) {
            attempts += a + 1;
            return true;
        }
        if (h < 0) {
            atomicOr(S.status, kErrHashFull);
            return false;
        }
    }
    attempts += S.max_attempts;
    atomicOr(S.status, kErrExhausted);
    return false;
}

// ------------------------------------------------- loss, fold, gradient out
// Fixed-order reduction of the block partials by one block of kThreads.
__device__ __forceinline__ void finish_loss_block(const LossSpec &l) {
    __shared__ double sh[3][kThreads];
    double t[3] = {0.0, 0.0, 0.0};
    for (int b = threadIdx.x; b < l.nblocks; b += kThreads)
        for (int c = 0; c < 3; ++c) t[c] += l.partials[4 * b + c];
    for (int c = 0; c < 3; ++c) sh[c][threadIdx.x] = t[c];
    __syncthreads();
    for (int w = kThreads / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int c = 0; c < 3; ++c) sh[c][threadIdx.x] += sh[c][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double loss = l.w_nz * sh[0][0] + l.w_z * sh[1][0];
        l.dloss[0] = loss;
        l.dloss[1] = sh[2][0];
        if (l.out) *l.out = loss;
        const int bits = isfinite(loss) ? 0 : kErrNonfinite;
        if (l.h_loss) {
            l.h_loss[0] = loss;
            l.h_loss[1] = sh[2][0];
            // every earlier kernel of the stream has set its bits; this one's
            // are the non-finite loss alone
            *l.h_status = atomicOr(l.status, bits) | bits;
        } else if (bits) {
            atomicOr(l.status, bits);
        }
    }
}

__global__ void __launch_bounds__(kThreads) k_finish_loss(const LossSpec l) {
    grid_wait();
    grid_trigger();
    finish_loss_block(l);
}

// Rows of Rp floats copied to rows of R, V columns per thread (V = 4 where R
// and the address of `out` allow 16-byte stores), by the first `nblocks`
// blocks; rows with a slot in `skip` (if given) are left out.
template <int V>
__device__ __forceinline__ void unpad_rows(const float *src, int Rp, int R, int64_t rows, float *out,
                                           const int *__restrict__ skip, int nblocks) {
    const unsigned units = (unsigned)(R / V);  // vectors or columns of a row
    const int64_t n = rows * units;            // below 2^31
    for (int64_t e = (int64_t)blockIdx.x * kThreads + threadIdx.x; e < n; e += (int64_t)nblocks * kThreads) {
        const unsigned row = (unsigned)e / units, u = (unsigned)e - row * units;
        if (skip && __ldg(skip + row) >= 0) continue;
        const float *g = src + (int64_t)row * Rp + V * u;
        if (V == 4)
            reinterpret_cast<float4 *>(out)[e] = *reinterpret_cast<const float4 *>(g);
        else
            out[e] = *g;
    }
}

// The epilogue of a gradient call after the fused pass, in one launch:
//  - the last block finishes the FP64 loss (and hands it to the caller's
//    device word or the pinned mirrors);
//  - with a caller's array, the first `ncold` blocks copy the rows of G that
//    have no replicas into its rows of R columns (unpad_rows);
//  - the blocks between take the quads of hot rows, one per group of NREP / 4
//    lanes: all replica quads of a hot quad are in flight at once
//    (gcpe::hot_quad_sum, which clears them for the next call), and the
//    group's first lane adds them to G (which may already hold contributions
//    of drawn cells to a replicated row of a large mode) and to the copy.
// Latency bound on small models, bandwidth bound on large ones.  It takes the
// place of a fold launch, a loss launch, a (strided) copy of the gradient,
// one of the loss and, for host results, two copies into pinned words: the
// smallest gradient call 32.2 -> 23.5 us, rank 50 on 172 x 25,000 x 300 at
// 2^16 samples 47.4 -> 30.2 us, rank 20 on 4999 x 3001 x 777 at 250,000
// samples 52.2 -> 41.0 us.
template <int NREP, int V>
__global__ void __launch_bounds__(kThreads) k_grad_finish(const GradOutSpec P, int ncold) {
    grid_wait();
    grid_trigger();
    if (blockIdx.x == gridDim.x - 1) {
        finish_loss_block(P.loss);
        return;
    }
    float4 *__restrict__ G4 = reinterpret_cast<float4 *>(P.G);
    if constexpr (NREP > 0) {
        if ((int)blockIdx.x >= ncold) {
            constexpr int H = gcpe::hot_lanes<NREP>();
            const int log2Q = __ffs(P.Rp) - 3;  // log2 of the quads of a row (Rp is a power of two)
            const int64_t hq = (int64_t)(blockIdx.x - ncold) * (kThreads / H) + (threadIdx.x / H);
            if (hq >= ((int64_t)P.Htot << log2Q)) return;  // the whole group leaves together
            const int slot = (int)(hq >> log2Q), cq = (int)(hq & ((1 << log2Q) - 1));
            const int row = __ldg(P.hot_row + slot);
            const int64_t q = ((int64_t)row << log2Q) + cq;
            const bool lead = (threadIdx.x & (H - 1)) == 0;
            float4 g;
            if (lead) g = G4[q];
            const float4 t = gcpe::hot_quad_sum<NREP>(
                reinterpret_cast<float4 *>(P.Grep + (int64_t)slot * P.rstride) + cq, P.rplane >> 2,
                gcpe::hot_group_mask<NREP>());
            if (!lead) return;
            g.x += t.x;
            g.y += t.y;
            g.z += t.z;
            g.w += t.w;
            G4[q] = g;
            if (!P.out) return;
            const int col = cq << 2;
            float *o = P.out + (int64_t)row * P.R + col;
            if (V == 4) {
                if (col < P.R) *reinterpret_cast<float4 *>(o) = g;
            } else {
                const float gv[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
                for (int j = 0; j < 4; ++j)
                    if (col + j < P.R) o[j] = gv[j];
            }
            return;
        }
    }
    unpad_rows<V>(P.G, P.Rp, P.R, P.rows, P.out, NREP > 0 ? P.hot_slot : nullptr, ncold);  // not the hot blocks' rows
}

// The same for a plain copy (factors out).
template <int V>
__global__ void __launch_bounds__(kThreads) k_unpad(const float *src, int Rp, int R, int64_t rows, float *out) {
    grid_wait();
    grid_trigger();
    unpad_rows<V>(src, Rp, R, rows, out, nullptr, gridDim.x);
}

// ------------------------------------------------------------- sampling
template <int D>
__global__ void __launch_bounds__(kThreads) k_sample(const SampleSpec S, int32_t *idx_out, float *x_out,
                                                    float *w_out, float w_nz, float w_z) {
    const int64_t n = S.p + S.q;
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < n; s += (int64_t)gridDim.x * blockDim.x) {
        int32_t idx[D];
        float x = 0.0f;
        int att = 0;
        draw_sample<D>(S, s, idx, x, att);
        if (idx_out)
#pragma unroll
            for (int k = 0; k < D; ++k) idx_out[s * D + k] = idx[k];
        if (x_out) x_out[s] = x;
        if (w_out) w_out[s] = s < S.p ? w_nz : w_z;
    }
}

// ------------------------------------------------------ nonzero records
__global__ void k_build_records(const int32_t *__restrict__ coords, const float *__restrict__ vals, int64_t nnz,
                                int d, SampleSpec S, RowOffsets ro, const int *__restrict__ hot_slot, int rec_words,
                                int32_t *rec, uint64_t *hkeys, uint64_t hbmask, int *status) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x) {
        uint64_t L = 0;
        int32_t *r = rec + e * rec_words;
        for (int k = d + 1; k < rec_words; ++k) r[k] = 0;
        for (int k = 0; k < d; ++k) {
            const int32_t c = coords[e * d + k];
            r[k] = c;
            L += (uint64_t)c * S.stride[k];
            const int hs = hot_slot ? hot_slot[ro.off[k] + c] : -1;
            const unsigned code = hs >= 0 ? (unsigned)hs : kNoSlot;
            r[d + 1 + k / 2] |= (int32_t)(code << (16 * (k & 1)));
        }
        r[d] = __float_as_int(vals[e]);
        const int rc = hash_insert(hkeys, hbmask, L);
        if (rc) atomicOr(status, rc);
    }
}

// ------------------------------------------------------------------ Adam
// Algorithm 1 on the flat parameter vector (Sec. 3.1.3); padded columns
// (col >= R) stay zero.  With BF16 storage the kernel-read copy is refreshed.
// Algorithm 1 on one 16-byte quad of parameters (columns col..col+3 of one
// row); padded columns (>= R) stay as they are (zero).  Abf, if not NULL,
// receives the BF16 copy of the quad.
__device__ __forceinline__ void adam_quad(float4 &a4, float4 &b4, float4 &c4, const float4 g4, int col, int R,
                                          float lr, float beta1, float beta2, float c1inv, float c2inv, float eps,
                                          float lower, uint2 *Abf) {
    float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w}, cv[4] = {c4.x, c4.y, c4.z, c4.w};
    const float gv[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (col + j >= R) continue;
        const float g = gv[j];
        bv[j] = beta1 * bv[j] + (1.0f - beta1) * g;
        cv[j] = beta2 * cv[j] + (1.0f - beta2) * g * g;
        av[j] = fmaxf(av[j] - lr * ((bv[j] * c1inv) / sqrtf(cv[j] * c2inv + eps)), lower);
    }
    a4 = make_float4(av[0], av[1], av[2], av[3]);
    b4 = make_float4(bv[0], bv[1], bv[2], bv[3]);
    c4 = make_float4(cv[0], cv[1], cv[2], cv[3]);
    if (Abf) {
        const __nv_bfloat162 lo = __floats2bfloat162_rn(av[0], av[1]), hi = __floats2bfloat162_rn(av[2], av[3]);
        *Abf = make_uint2(*reinterpret_cast<const unsigned *>(&lo), *reinterpret_cast<const unsigned *>(&hi));
    }
}

// Algorithm 1 over the flat parameter vector, one quad per thread and step
// (n and Rp are multiples of 4, Rp a power of two, so a quad is in one row).
__global__ void k_adam(int64_t n, int Rp, int R, float *__restrict__ A, float *__restrict__ B,
                       float *__restrict__ C, const float *__restrict__ G, float lr, float beta1, float beta2,
                       float c1inv, float c2inv, float eps, float lower, __nv_bfloat16 *Abf) {
    for (int64_t qi = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; qi < (n >> 2);
         qi += (int64_t)gridDim.x * blockDim.x) {
        const int col = (int)((qi << 2) & (Rp - 1));
        if (col >= R) continue;
        float4 a4 = reinterpret_cast<const float4 *>(A)[qi], b4 = reinterpret_cast<const float4 *>(B)[qi],
               c4 = reinterpret_cast<const float4 *>(C)[qi];
        adam_quad(a4, b4, c4, reinterpret_cast<const float4 *>(G)[qi], col, R, lr, beta1, beta2, c1inv, c2inv, eps,
                  lower, Abf ? reinterpret_cast<uint2 *>(Abf) + qi : nullptr);
        reinterpret_cast<float4 *>(A)[qi] = a4;
        reinterpret_cast<float4 *>(B)[qi] = b4;
        reinterpret_cast<float4 *>(C)[qi] = c4;
    }
}

// One training step's epilogue after the fused pass, in one launch, on
// 16-byte quads of the flat parameter vector (Rp is a power of two and a
// multiple of 4, so a quad lies in one row):
//  - the last block finishes the FP64 loss from the block partials (fixed
//    order);
//  - the first `ncold` blocks stream the quads of rows without replicas:
//    each thread takes kPostUnroll quads per iteration and issues all of
//    their loads (gradient, moments, factor, replica slot) before using any,
//    then applies Algorithm 1 and clears G for the next step;
//  - the blocks between take the quads of hot rows, one per group of
//    NREP / 4 lanes: the group loads the quad's NREP replica quads at
//    once (gcpe::hot_quad_sum, which also clears them), and its first lane
//    adds them to the gradient quad and applies Algorithm 1.  With NREP = 0
//    there are no hot rows and no such blocks.
// The streaming blocks run at the copy rate on models larger than L2; the
// hot quads cost one memory round trip each instead of one per group of
// replica loads.
// Quads per streaming thread and iteration, and waves of resident streaming
// blocks at most.  One quad per thread streamed the HBM-resident epilogue
// (121.6M parameters) at 6.0 TB/s; two or four per thread, with fewer
// resident warps, at 3.6 and 4.1 TB/s.  With one wave of blocks striding over
// the arrays the rate hangs on how the eight streams fall on the memory
// banks: a step of that model took 2.77, 2.31, 2.22, 2.27 and 2.24 ms on 304,
// 608, 700, 760 and 912 blocks, and 4.2 ms when the compiler chose a few
// registers more; with 13 to 40 waves, which the hardware hands out as blocks
// finish, 2.14 ms (the epilogue at 6.6 TB/s).
constexpr int kPostUnroll = 1;
constexpr int kPostWaves = 16;

template <int NREP>
__global__ void __launch_bounds__(kThreads) k_post_step(PostSpec P, int ncold) {
    grid_wait();
    grid_trigger();  // the next step's pass may draw its samples beside this grid
    if (blockIdx.x == gridDim.x - 1) {  // the last block only finishes the loss
        finish_loss_block(P.loss);
        return;
    }
    float4 *__restrict__ G4 = reinterpret_cast<float4 *>(P.G);
    float4 *__restrict__ A4 = reinterpret_cast<float4 *>(P.A);
    float4 *__restrict__ B4 = reinterpret_cast<float4 *>(P.B);
    float4 *__restrict__ C4 = reinterpret_cast<float4 *>(P.C);
    uint2 *__restrict__ Abf = static_cast<uint2 *>(P.Abf);
    const int log2Rp = __ffs(P.Rp) - 1;
    if constexpr (NREP > 0) {
        if ((int)blockIdx.x >= ncold) {  // hot quads, one per group of NREP / 4 lanes
            constexpr int H = gcpe::hot_lanes<NREP>();
            const int log2Q = log2Rp - 2;  // quads per row = Rp / 4
            const int64_t hq = (int64_t)(blockIdx.x - ncold) * (kThreads / H) + (threadIdx.x / H);
            if (hq >= ((int64_t)P.Htot << log2Q)) return;  // the whole group leaves together
            const int slot = (int)(hq >> log2Q), cq = (int)(hq & ((1 << log2Q) - 1));
            const int64_t q = ((int64_t)__ldg(P.hot_row + slot) << log2Q) + cq;
            const bool lead = (threadIdx.x & (H - 1)) == 0;
            float4 g, a, b, c;
            if (lead) {
                g = G4[q];
                a = A4[q];
                b = B4[q];
                c = C4[q];
            }
            const float4 t = gcpe::hot_quad_sum<NREP>(
                reinterpret_cast<float4 *>(P.Grep + (int64_t)slot * P.rstride) + cq, P.rplane >> 2,
                gcpe::hot_group_mask<NREP>());
            if (!lead) return;
            g.x += t.x;
            g.y += t.y;
            g.z += t.z;
            g.w += t.w;
            G4[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            const int col = cq << 2;
            if (col >= P.R) return;  // a quad of padding columns
            adam_quad(a, b, c, g, col, P.R, P.lr, P.beta1, P.beta2, P.c1inv, P.c2inv, P.eps, P.lower,
                      Abf ? Abf + q : nullptr);
            A4[q] = a;
            B4[q] = b;
            C4[q] = c;
            return;
        }
    }
    // block tiles of kThreads * kPostUnroll consecutive quads; thread t takes
    // quads t, t + kThreads, ... of its block's tile
    const int64_t nq = P.n >> 2;
    constexpr int64_t kTile = (int64_t)kThreads * kPostUnroll;
    for (int64_t q0 = (int64_t)blockIdx.x * kTile + threadIdx.x; q0 < nq; q0 += (int64_t)ncold * kTile) {
        float4 g[kPostUnroll], a[kPostUnroll], b[kPostUnroll], c[kPostUnroll];
        int hs[kPostUnroll];
#pragma unroll
        for (int u = 0; u < kPostUnroll; ++u) {
            const int64_t q = q0 + u * kThreads;
            hs[u] = -1;
            if (q < nq) {
                g[u] = G4[q];
                a[u] = A4[q];
                b[u] = B4[q];
                c[u] = C4[q];
                if (P.hot_slot) hs[u] = __ldg(P.hot_slot + ((q << 2) >> log2Rp));
            }
        }
#pragma unroll
        for (int u = 0; u < kPostUnroll; ++u) {
            const int64_t q = q0 + u * kThreads;
            if (q >= nq || hs[u] >= 0) continue;  // hot quads belong to the hot blocks
            G4[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            const int col = (int)((q << 2) & (P.Rp - 1));
            if (col >= P.R) continue;  // a quad of padding columns: nothing to update
            adam_quad(a[u], b[u], c[u], g[u], col, P.R, P.lr, P.beta1, P.beta2, P.c1inv, P.c2inv, P.eps, P.lower,
                      Abf ? Abf + q : nullptr);
            A4[q] = a[u];
            B4[q] = b[u];
            C4[q] = c[u];
        }
    }
}

template <int NREP>
static cudaError_t launch_post_step_r(const PostSpec &p, cudaStream_t st) {
    static int resident = 0;  // streaming blocks that fit on the GPU at once
    if (!resident) {
        int per_sm = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_post_step<NREP>, kThreads, 0);
        resident = (per_sm < 1 ? 1 : per_sm) * num_sms();
    }
    const int64_t want = ((p.n >> 2) + (int64_t)kThreads * kPostUnroll - 1) / ((int64_t)kThreads * kPostUnroll);
    const int64_t cap = (int64_t)kPostWaves * resident;
    const int ncold = (int)(want < 1 ? 1 : (want > cap ? cap : want));
    int nhot = 0;
    if constexpr (NREP > 0) {
        constexpr int per = kThreads / gcpe::hot_lanes<NREP>();  // hot quads of a block
        nhot = (int)(((int64_t)p.Htot * (p.Rp >> 2) + per - 1) / per);
    }
    const int blocks = ncold + nhot + 1;  // + the loss block
    return launch_dependent(k_post_step<NREP>, blocks, kThreads, 0, st, p, ncold);
}

cudaError_t launch_post_step(const PostSpec &p, cudaStream_t st) {
    switch (p.nrep) {
    case 0: return launch_post_step_r<0>(p, st);
    case 4: return launch_post_step_r<4>(p, st);
    case 16: return launch_post_step_r<16>(p, st);
    case 64: return launch_post_step_r<64>(p, st);
    default: return cudaErrorInvalidValue;
    }
}

__global__ void k_to_bf16(int64_t n, const float *__restrict__ A, __nv_bfloat16 *Abf) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
        Abf[e] = __float2bfloat16_rn(A[e]);
}

// --------------------------------------------------------------- launches
static int elementwise_blocks(int64_t n) {
    const int64_t want = (n + kThreads - 1) / kThreads;
    const int64_t cap = (int64_t)num_sms() * 8;
    return (int)(want < 1 ? 1 : (want > cap ? cap : want));
}

cudaError_t launch_build_records(const int32_t *coords, const float *vals, int64_t nnz, int d,
                                 const uint64_t *stride, const int64_t *rowoff, const int *hot_slot,
                                 int rec_words, int32_t *rec, uint64_t *hkeys, uint64_t hbmask, int *status,
                                 cudaStream_t st) {
    SampleSpec S{};
    S.d = d;
    RowOffsets ro{};
    for (int k = 0; k < d; ++k) {
        S.stride[k] = stride[k];
        ro.off[k] = rowoff[k];
    }
    k_build_records<<<elementwise_blocks(nnz), kThreads, 0, st>>>(coords, vals, nnz, d, S, ro, hot_slot, rec_words,
                                                                   rec, hkeys, hbmask, status);
    return cudaGetLastError();
}

#define GCP_DISPATCH_D(d, MACRO) \
    switch (d) {                 \
    case 2: MACRO(2); break;     \
    case 3: MACRO(3); break;     \
    case 4: MACRO(4); break;     \
    case 5: MACRO(5); break;     \
    case 6: MACRO(6); break;     \
    case 7: MACRO(7); break;     \
    case 8: MACRO(8); break;     \
    default: return cudaErrorInvalidValue; \
    }

cudaError_t launch_sample(const SampleSpec &s, int32_t *idx_out, float *x_out, float *w_out, float w_nz,
                          float w_z, cudaStream_t st) {
    const int64_t n = s.p + s.q;
    if (n == 0) return cudaSuccess;
    const int blocks = elementwise_blocks(n);
#define GCP_LAUNCH_SAMPLE(D) k_sample<D><<<blocks, kThreads, 0, st>>>(s, idx_out, x_out, w_out, w_nz, w_z)
    GCP_DISPATCH_D(s.d, GCP_LAUNCH_SAMPLE)
#undef GCP_LAUNCH_SAMPLE
    return cudaGetLastError();
}

// Non-fused MTTKRP (Sec. 3.1.2 before fusion): reads the gradient tensor the
// sampling pass wrote (cells Ycoord, values Yval), gathers the factor rows
// again and adds y prod_{k!=n} A_k(i_k,:) to every mode's rows, with the
// same hot-row replicas as the fused pass (slots looked up by row).
template <int D, typename TF, int COLS>
__global__ void __launch_bounds__(kThreads) k_mttkrp_nonfused(const FusedSpec P, const int *__restrict__ hot_slot,
                                                             int S) {
    constexpr int NQ = COLS / 4;
    const int lane = threadIdx.x & 31;
    const int L = 1 << P.log2L;
    const int glane = lane & (L - 1);
    const int group = (blockIdx.x * blockDim.x + threadIdx.x) >> P.log2L;
    const int ngroups = (gridDim.x * blockDim.x) >> P.log2L;
    const int warp0 = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const TF *__restrict__ F = static_cast<const TF *>(P.F);
    float *const grep = P.Grep ? P.Grep + (size_t)(warp0 & (P.nrep - 1)) * P.rplane : nullptr;
    int col[NQ];
    bool on[NQ];  // the quad holds columns of the rank, not padding alone
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        col[q] = q * (P.Rp >> 1) + 4 * glane;
        on[q] = col[q] < P.R;
    }
    for (int s = group; s < S; s += ngroups) {
        const float y = __ldg(P.Yval + (int64_t)s * P.vstride);
        int ii[D], off[D];
        float a[D][COLS];
#pragma unroll
        for (int k = 0; k < D; ++k) {
            ii[k] = __ldg(P.Ycoord + (int64_t)s * P.ystride + k);
            off[k] = (P.rowoff[k] + ii[k]) * P.Rp;
#pragma unroll
            for (int q = 0; q < NQ; ++q) Quad<TF>::load(F + off[k] + col[q], a[k] + 4 * q);
        }
        float suf[D][COLS];
#pragma unroll
        for (int v = 0; v < COLS; ++v) suf[D - 1][v] = 1.0f;
#pragma unroll
        for (int k = D - 2; k >= 0; --k)
#pragma unroll
            for (int v = 0; v < COLS; ++v) suf[k][v] = suf[k + 1][v] * a[k + 1][v];
        float pre[COLS];
#pragma unroll
        for (int v = 0; v < COLS; ++v) pre[v] = y;
#pragma unroll
        for (int n = 0; n < D; ++n) {
            const int hs = hot_slot ? __ldg(hot_slot + P.rowoff[n] + ii[n]) : -1;
            float *g = hs >= 0 ? grep + hs * P.rstride : P.G + off[n];
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

template <int D>
static void launch_nonfused_d(const FusedSpec &f, const int *hot_slot, int S, bool bf16, int cols, int blocks,
                              cudaStream_t st) {
    if (bf16) {
        if (cols == 8)
            k_mttkrp_nonfused<D, __nv_bfloat16, 8><<<blocks, kThreads, 0, st>>>(f, hot_slot, S);
        else
            k_mttkrp_nonfused<D, __nv_bfloat16, 4><<<blocks, kThreads, 0, st>>>(f, hot_slot, S);
    } else {
        if (cols == 8)
            k_mttkrp_nonfused<D, float, 8><<<blocks, kThreads, 0, st>>>(f, hot_slot, S);
        else
            k_mttkrp_nonfused<D, float, 4><<<blocks, kThreads, 0, st>>>(f, hot_slot, S);
    }
}

cudaError_t launch_mttkrp_nonfused(const FusedSpec &f, const int *hot_slot, bool bf16, int cols, int max_blocks,
                                   cudaStream_t st) {
    const int S = (int)(f.s.p + f.s.q);
    if (S == 0) return cudaSuccess;
    const int64_t lanes = (int64_t)S << f.log2L;
    int64_t want = (lanes + kThreads - 1) / kThreads;
    const int blocks = (int)(want < max_blocks ? (want < 1 ? 1 : want) : max_blocks);
    switch (f.s.d) {
    case 2: launch_nonfused_d<2>(f, hot_slot, S, bf16, cols, blocks, st); break;
    case 3: launch_nonfused_d<3>(f, hot_slot, S, bf16, cols, blocks, st); break;
    case 4: launch_nonfused_d<4>(f, hot_slot, S, bf16, cols, blocks, st); break;
    case 5: launch_nonfused_d<5>(f, hot_slot, S, bf16, cols, blocks, st); break;
    case 6: launch_nonfused_d<6>(f, hot_slot, S, bf16, cols, blocks, st); break;
    case 7: launch_nonfused_d<7>(f, hot_slot, S, bf16, cols, blocks, st); break;
    case 8: launch_nonfused_d<8>(f, hot_slot, S, bf16, cols, blocks, st); break;
    default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
}

template <int NREP, int V>
static cudaError_t launch_grad_finish_rv(const GradOutSpec &p, cudaStream_t st) {
    const int ncold = p.out ? elementwise_blocks(p.rows * (p.R / V)) : 0;
    int nhot = 0;
    if constexpr (NREP > 0) {
        constexpr int per = kThreads / gcpe::hot_lanes<NREP>();  // hot quads of a block
        nhot = (int)(((int64_t)p.Htot * (p.Rp >> 2) + per - 1) / per);
    }
    const int blocks = ncold + nhot + 1;  // + the loss block
    return launch_dependent(k_grad_finish<NREP, V>, blocks, kThreads, 0, st, p, ncold);
}

template <int NREP>
static cudaError_t launch_grad_finish_r(const GradOutSpec &p, cudaStream_t st) {
    const bool vec = p.R % 4 == 0 && (reinterpret_cast<uintptr_t>(p.out) & 15) == 0;
    return vec ? launch_grad_finish_rv<NREP, 4>(p, st) : launch_grad_finish_rv<NREP, 1>(p, st);
}

cudaError_t launch_grad_finish(const GradOutSpec &p, cudaStream_t st) {
    switch (p.nrep) {
    case 0: return launch_grad_finish_r<0>(p, st);
    case 4: return launch_grad_finish_r<4>(p, st);
    case 16: return launch_grad_finish_r<16>(p, st);
    case 64: return launch_grad_finish_r<64>(p, st);
    default: return cudaErrorInvalidValue;
    }
}

cudaError_t launch_finish_loss(const LossSpec &l, cudaStream_t st) {
    return launch_dependent(k_finish_loss, 1, kThreads, 0, st, l);
}

cudaError_t launch_unpad(const float *src, int Rp, int R, int64_t rows, float *out, cudaStream_t st) {
    if (R % 4 == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0)
        return launch_dependent(k_unpad<4>, elementwise_blocks(rows * (R / 4)), kThreads, 0, st, src, Rp, R, rows, out);
    return launch_dependent(k_unpad<1>, elementwise_blocks(rows * R), kThreads, 0, st, src, Rp, R, rows, out);
}

// x = 0 before a gradient pass, as a kernel and not a memset so that the pass
// may start beside it.
__global__ void __launch_bounds__(kThreads) k_clear(float4 *x, int64_t nq) {
    grid_wait();
    grid_trigger();
    for (int64_t q = (int64_t)blockIdx.x * kThreads + threadIdx.x; q < nq; q += (int64_t)gridDim.x * kThreads)
        x[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
}

cudaError_t launch_clear(float *x, int64_t n, cudaStream_t st) {
    return launch_dependent(k_clear, elementwise_blocks(n >> 2), kThreads, 0, st, reinterpret_cast<float4 *>(x), n >> 2);
}

cudaError_t launch_adam(int64_t n, int Rp, int R, float *A, float *B, float *C, const float *G, float lr,
                        float beta1, float beta2, float c1inv, float c2inv, float eps, float lower, void *Abf,
                        cudaStream_t st) {
    // many blocks per SM, as in k_post_step: 121.6M parameters 540 -> 496 us
    const int64_t want = ((n >> 2) + kThreads - 1) / kThreads, cap = (int64_t)num_sms() * 64;
    k_adam<<<(int)(want < 1 ? 1 : (want < cap ? want : cap)), kThreads, 0, st>>>(n, Rp, R, A, B, C, G, lr, beta1, beta2, c1inv, c2inv, eps,
                                                        lower, static_cast<__nv_bfloat16 *>(Abf));
    return cudaGetLastError();
}

cudaError_t launch_to_bf16(int64_t n, const float *A, void *Abf, cudaStream_t st) {
    k_to_bf16<<<elementwise_blocks(n), kThreads, 0, st>>>(n, A, static_cast<__nv_bfloat16 *>(Abf));
    return cudaGetLastError();
}

}  // namespace gcpk
