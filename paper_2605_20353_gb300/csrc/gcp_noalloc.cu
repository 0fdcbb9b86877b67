// gcp_noalloc.cu -- sampled GCP loss and gradient of a caller-supplied
// sample list, without any device allocation.
//
// Some callers cannot allocate device memory: code that runs under a device
// memory budget fixed when it starts (a host framework that owns every
// allocation through its own pool, or a long-running service that must not
// grow its footprint after start-up).  This entry point takes all of its
// inputs and outputs from the caller and keeps its only scratch -- one loss
// partial per block -- in the file-scope device array below.  That array is
// part of the library image: every GPU that loads the library holds it
// (8192 slots x 16 bytes = 128 KB) until the
// process exits.
#include <algorithm>
#include <mutex>

#include "../../include/gcp.h"
#include "gcp_device.cuh"
#include "gcp_internal.h"

using namespace gcpdev;

namespace {

constexpr int kNaThreads = 256;
constexpr int kNaWarps = kNaThreads / 32;
constexpr int kNaMaxBlocks = 8192;
constexpr int kNaMaxDevices = 64;

// Per-block (loss partial, skipped-sample count), shared by every call on a
// device.  Each call writes the slots of the blocks it launches before it
// reads them, so nothing has to start at zero; calls that overlap on the
// GPU race on these slots.
__device__ __align__(256) double2 g_na_partials[kNaMaxBlocks];

struct NaShape {
    int R;
    int log2L;                       // lanes per sample
    int64_t dims[GCP_MAX_NDIM];
    int64_t rowoff[GCP_MAX_NDIM];
};

// V consecutive columns of a row of A, or added to a row of G: one 16-byte
// vector (V = 4) or a scalar (V = 1).
template <int V>
__device__ __forceinline__ void na_load(const float *p, float *o) {
    if (V == 4)
        Quad<float>::load(p, o);
    else
        o[0] = __ldg(p);
}
template <int V>
__device__ __forceinline__ void na_add(float *p, const float *c) {
    if (V == 4)
        red_add_v4(p, c[0], c[1], c[2], c[3]);
    else
        atomicAdd(p, c[0]);
}

// Sampled gradient of a sample list.  A warp takes tiles of 32 consecutive
// samples: lane l reads sample l's coordinates, value and weight (the next
// tile's are in flight while this one is evaluated), then groups of L lanes
// take the tile's samples in turn, their row offsets, values and weights
// handed over by shuffles.  Lane g of a group owns columns V (g + L q) ..
// V (g + L q) + V - 1 for q < NQ; those past the rank are skipped, so rows
// need no padding.  Each lane keeps its own sample's loss and adds it in
// FP64 once per tile (three FP64 instructions per 32 samples).
// Bound by the row traffic through L2 (d rows gathered, d rows reduced per
// sample) and, on skewed data, by the reductions that meet in one row: the
// entry point has no scratch for replicas.  2^18 samples of the 2000 x 1500
// x 1000 x 200 Zipf tensor at rank 32, drawn with gcp_sample and passed
// here: 156 us a pass, against 745 us with one warp per sample walking 256
// samples one after another on 128 blocks.
template <int D, int V, int NQ>
__global__ void __launch_bounds__(kNaThreads, (D <= 4 ? 3 : 1))
    k_na_grad(const NaShape sh, int loss, int64_t n, const int32_t *__restrict__ idx, const float *__restrict__ x,
              const float *__restrict__ w, const float *__restrict__ A, float *__restrict__ G, double2 *partials) {
    constexpr int C = V * NQ;  // columns per lane
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int L = 1 << sh.log2L;
    const int glane = lane & (L - 1), grp = lane >> sh.log2L, ngrp = 32 >> sh.log2L;
    int col[NQ];
    bool on[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
        col[q] = V * (glane + L * q);
        on[q] = col[q] < sh.R;
    }
    const int64_t ntiles = (n + 31) >> 5;
    const int64_t nwarps = (int64_t)gridDim.x * kNaWarps;
    int32_t ni[D];  // the next tile's sample of this lane
    float nx = 0.0f, nw = 0.0f;
    auto fetch = [&](int64_t tile) {
        const int64_t s = (tile << 5) + lane;
        if (s < n) {
#pragma unroll
            for (int k = 0; k < D; ++k) ni[k] = __ldg(idx + s * D + k);
            nx = __ldg(x + s);
            nw = __ldg(w + s);
        } else {
#pragma unroll
            for (int k = 0; k < D; ++k) ni[k] = 0;
        }
    };
    double acc = 0.0;
    int skipped = 0;
    int64_t tile = (int64_t)blockIdx.x * kNaWarps + warp;
    fetch(tile);
    for (; tile < ntiles; tile += nwarps) {
        bool ok = true;
        int64_t row[D];
#pragma unroll
        for (int k = 0; k < D; ++k) {
            ok = ok && ni[k] >= 0 && ni[k] < sh.dims[k];
            row[k] = (sh.rowoff[k] + ni[k]) * sh.R;
        }
        const float myx = nx, myw = nw;
        const bool in = (tile << 5) + lane < n;
        skipped += in && !ok;  // out-of-range coordinates: the sample is skipped and counted
        const unsigned okmask = __ballot_sync(0xFFFFFFFFu, in && ok);
        fetch(tile + nwarps);
        float myf = 0.0f;
        for (int it = 0; it < L; ++it) {
            const int src = it * ngrp + grp;
            const bool live = (okmask >> src) & 1u;  // uniform within the group
            const float xs = __shfl_sync(0xFFFFFFFFu, myx, src), ws = __shfl_sync(0xFFFFFFFFu, myw, src);
            int64_t off[D];
            float a[D][C];
#pragma unroll
            for (int k = 0; k < D; ++k) {
                off[k] = __shfl_sync(0xFFFFFFFFu, row[k], src);
#pragma unroll
                for (int v = 0; v < C; ++v) a[k][v] = 0.0f;
            }
            if (live)
#pragma unroll
                for (int k = 0; k < D; ++k)
#pragma unroll
                    for (int q = 0; q < NQ; ++q)
                        if (on[q]) na_load<V>(A + off[k] + col[q], a[k] + V * q);
            float suf[D][C];  // suf[k] = prod_{j>k} a_j
#pragma unroll
            for (int v = 0; v < C; ++v) suf[D - 1][v] = 1.0f;
#pragma unroll
            for (int k = D - 2; k >= 0; --k)
#pragma unroll
                for (int v = 0; v < C; ++v) suf[k][v] = suf[k + 1][v] * a[k + 1][v];
            float m = 0.0f;
#pragma unroll
            for (int v = 0; v < C; ++v) m = fmaf(a[0][v], suf[0][v], m);
            for (int o = L >> 1; o > 0; o >>= 1) m += __shfl_xor_sync(0xFFFFFFFFu, m, o);
            float f, df;
            loss_eval(loss, xs, m, f, df);
            // sample `lane` was evaluated by group lane % ngrp in round lane / ngrp
            const float fl = __shfl_sync(0xFFFFFFFFu, f, (lane & (ngrp - 1)) << sh.log2L);
            if ((lane >> (5 - sh.log2L)) == it) myf = fl;
            if (!live) continue;
            float pre[C];
#pragma unroll
            for (int v = 0; v < C; ++v) pre[v] = ws * df;
#pragma unroll
            for (int k = 0; k < D; ++k) {
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    if (!on[q]) continue;
                    float c[V];
#pragma unroll
                    for (int v = 0; v < V; ++v) c[v] = pre[V * q + v] * suf[k][V * q + v];
                    na_add<V>(G + off[k] + col[q], c);
                }
#pragma unroll
                for (int v = 0; v < C; ++v) pre[v] *= a[k][v];
            }
        }
        __syncwarp();
        if ((okmask >> lane) & 1u) acc += (double)myw * (double)myf;
    }
    // block partial: a fixed butterfly over the lanes, then the warps in order
    double sk = (double)skipped;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
        sk += __shfl_xor_sync(0xFFFFFFFFu, sk, o);
    }
    __shared__ double2 red[kNaWarps];
    if (lane == 0) red[warp] = make_double2(acc, sk);
    __syncthreads();
    if (threadIdx.x == 0) {
        double2 t = make_double2(0.0, 0.0);
        for (int i = 0; i < kNaWarps; ++i) {
            t.x += red[i].x;
            t.y += red[i].y;
        }
        partials[blockIdx.x] = t;
    }
}

// Fixed-order sum of the block partials: loss_out[0] = loss,
// loss_out[1] = samples skipped for out-of-range coordinates.
__global__ void __launch_bounds__(kNaThreads) k_na_sum(const double2 *partials, int nblocks, double *loss_out) {
    __shared__ double2 sh[kNaThreads];
    double2 t = make_double2(0.0, 0.0);
    for (int b = threadIdx.x; b < nblocks; b += kNaThreads) {
        t.x += partials[b].x;
        t.y += partials[b].y;
    }
    sh[threadIdx.x] = t;
    __syncthreads();
    for (int h = kNaThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            sh[threadIdx.x].x += sh[threadIdx.x + h].x;
            sh[threadIdx.x].y += sh[threadIdx.x + h].y;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        loss_out[0] = sh[0].x;
        loss_out[1] = sh[0].y;
    }
}

// Columns per lane and lanes per sample.  Vectors need a rank that is a
// multiple of 4 and 16-byte aligned A and G (every row then starts on a
// 16-byte boundary); other calls add one column at a time, a lane's columns
// L apart so that a group's reduction covers consecutive floats.
struct NaPlan {
    int v, nq, log2L;
};

NaPlan na_plan(int R, bool aligned) {
    NaPlan p{};
    p.v = (R % 4 == 0 && aligned) ? 4 : 1;
    const int units = R / p.v;  // vectors or columns of a row, at most 32 or 128
    p.nq = p.v == 4 ? (units > 8 ? 2 : 1) : (units > 64 ? 4 : (units > 16 ? 2 : 1));
    while ((p.nq << p.log2L) < units) ++p.log2L;
    return p;
}

using NaKernel = void (*)(NaShape, int, int64_t, const int32_t *, const float *, const float *, const float *, float *,
                          double2 *);

template <int D>
NaKernel na_kernel_d(const NaPlan &p) {
    if (p.v == 4) return p.nq == 2 ? k_na_grad<D, 4, 2> : k_na_grad<D, 4, 1>;
    return p.nq == 4 ? k_na_grad<D, 1, 4> : (p.nq == 2 ? k_na_grad<D, 1, 2> : k_na_grad<D, 1, 1>);
}

NaKernel na_kernel(int d, const NaPlan &p) {
    switch (d) {
    case 2: return na_kernel_d<2>(p);
    case 3: return na_kernel_d<3>(p);
    case 4: return na_kernel_d<4>(p);
    case 5: return na_kernel_d<5>(p);
    case 6: return na_kernel_d<6>(p);
    case 7: return na_kernel_d<7>(p);
    default: return na_kernel_d<8>(p);
    }
}

// Device address of g_na_partials, looked up once per device.  In host
// code the array's name is only a host-side stand-in, so the kernel must be
// given the address that cudaGetSymbolAddress returns for the current
// device.
std::mutex g_na_mutex;
double2 *g_na_addr[kNaMaxDevices] = {nullptr};

cudaError_t scratch_for_current_device(double2 **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kNaMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_na_partials);
        if (e != cudaSuccess) return e;
        g_na_addr[dev] = static_cast<double2 *>(p);
    }
    *out = g_na_addr[dev];
    return cudaSuccess;
}

gcp_status na_fail(gcp_status s, const char *msg) {
    gcpk_set_noctx_error(msg);  // read back with gcp_last_error(NULL)
    return s;
}

}  // namespace

extern "C" gcp_status gcp_grad_samples_noalloc(int32_t ndim, const int64_t *dims, int32_t rank, int32_t loss,
                                               int64_t nsamples, const int32_t *idx, const float *x, const float *w,
                                               const float *A, float *G, double *loss_out, void *stream) {
    if (ndim < 2 || ndim > GCP_MAX_NDIM || !dims) return na_fail(GCP_ERR_ARG, "ndim must be in 2..8");
    if (rank < 1 || rank > GCP_MAX_RANK) return na_fail(GCP_ERR_ARG, "rank must be in 1..128");
    if (loss < GCP_GAUSSIAN || loss > GCP_GAMMA) return na_fail(GCP_ERR_ARG, "unknown loss");
    if (nsamples < 0) return na_fail(GCP_ERR_ARG, "nsamples < 0");
    if (nsamples > GCP_NOALLOC_MAX_SAMPLES)
        return na_fail(GCP_ERR_ARG, "nsamples exceeds GCP_NOALLOC_MAX_SAMPLES (16777216), the capacity of this "
                                    "entry point's fixed scratch; split the samples over several calls");
    if (!A || !G || !loss_out || (nsamples > 0 && (!idx || !x || !w)))
        return na_fail(GCP_ERR_ARG, "NULL device pointer");
    const bool aligned = ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(G)) & 15) == 0;
    const NaPlan plan = na_plan(rank, aligned);
    NaShape sh{};
    sh.R = rank;
    sh.log2L = plan.log2L;
    int64_t rows = 0;
    for (int k = 0; k < ndim; ++k) {
        if (dims[k] < 1 || dims[k] > INT32_MAX) return na_fail(GCP_ERR_ARG, "mode size out of range");
        sh.dims[k] = dims[k];
        sh.rowoff[k] = rows;
        rows += dims[k];
    }
    double2 *scratch = nullptr;
    cudaError_t e = scratch_for_current_device(&scratch);
    if (e != cudaSuccess) return na_fail(GCP_ERR_CUDA, cudaGetErrorString(e));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if ((e = cudaMemsetAsync(G, 0, (size_t)rows * rank * sizeof(float), st)) != cudaSuccess)
        return na_fail(GCP_ERR_CUDA, cudaGetErrorString(e));
    int nblocks = 0;
    if (nsamples > 0) {
        // a grid of at most the blocks that fit on the GPU at once; fewer
        // when there are fewer tiles than warps
        const NaKernel k = na_kernel(ndim, plan);
        int dev = 0, sms = 0, per_sm = 0;
        if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
            (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
            (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kNaThreads, 0)) != cudaSuccess)
            return na_fail(GCP_ERR_CUDA, cudaGetErrorString(e));
        const int64_t want = ((nsamples + 31) / 32 + kNaWarps - 1) / kNaWarps;
        nblocks = (int)std::min<int64_t>(want, std::min<int64_t>((int64_t)std::max(1, per_sm) * sms, kNaMaxBlocks));
        k<<<nblocks, kNaThreads, 0, st>>>(sh, loss, nsamples, idx, x, w, A, G, scratch);
    }
    k_na_sum<<<1, kNaThreads, 0, st>>>(scratch, nblocks, loss_out);
    if ((e = cudaGetLastError()) != cudaSuccess) return na_fail(GCP_ERR_CUDA, cudaGetErrorString(e));
    return GCP_OK;
}
