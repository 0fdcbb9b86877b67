// gcp_noalloc.cu -- sampled GCP loss and gradient of a caller-supplied
// sample list, without any device allocation.
//
// Some callers cannot allocate device memory: code that runs under a device
// memory budget fixed when it starts (a host framework that owns every
// allocation through its own pool, or a long-running service that must not
// grow its footprint after start-up).  This entry point takes all of its
// inputs and outputs from the caller and keeps its only scratch -- one loss
// partial per block and a few replicas of the hottest gradient rows -- in the
// file-scope device array below.  That array is part of the library image:
// every GPU that loads the library holds it (128 KB) until the process exits.
//
// Three launches: the gradient cleared and the hot rows of the list found
// (k_na_setup), the pass over the samples (k_na_grad), the replicas folded and
// the loss summed (k_na_finish).
#include <algorithm>
#include <mutex>

#include "../../include/gcp.h"
#include "gcp_device.cuh"
#include "gcp_internal.h"
#include "gcp_noalloc_hot.h"

using namespace gcpdev;

namespace {

constexpr int kNaThreads = 256;
constexpr int kNaWarps = kNaThreads / 32;
constexpr int kNaMaxBlocks = 2048;
constexpr int kNaMaxDevices = 64;

// The hot rows of one mode: how many, with how many replicas each
// (gcpna::hot_word), and which.
struct NaHot {
    int word;
    int row[gcpna::kHot];
};

// Everything a call keeps on the device, shared by every call on it: loss
// partials (block loss, skipped samples), the hot rows, their replicas.  Each
// call writes what it reads later, so nothing has to start at zero; calls
// that overlap on the GPU race on it, and what a kernel finds is held to its
// own call's shape before it is used (gcp_noalloc_hot.h).
struct NaScratch {
    double2 partials[kNaMaxBlocks];
    NaHot hot[GCP_MAX_NDIM];
    alignas(16) float rep[gcpna::kRepFloats];
};
static_assert(sizeof(NaScratch) <= 128 * 1024, "the documented size of the scratch");
__device__ __align__(256) unsigned char g_na_scratch[128 * 1024];

struct NaShape {
    int R;
    int log2L;                       // lanes per sample
    int d;
    int hot;                         // whether the list is searched for hot rows
    int tile;                        // samples per warp tile (fused_tile)
    int64_t rows;
    int64_t dims[GCP_MAX_NDIM];
    int64_t rowoff[GCP_MAX_NDIM];
};

// Blocks k < d (if sh.hot): the hot rows of mode k.  kNaProbe samples spread
// over the list are counted in a hash table; the rows counted at least T times
// are hot, T the smallest of 8, 16, 32, ... with which there are at most
// kHot of them and four replicas of each fit the mode's share.  (A row that
// takes 1/256 of the samples is counted 8 times.)  The mode's replicas are
// cleared.  The other blocks clear G.
constexpr int kNaProbe = 2048, kNaTable = 4096;

__global__ void __launch_bounds__(kNaThreads) k_na_setup(const NaShape sh, int64_t n, const int32_t *__restrict__ idx,
                                                        float *__restrict__ G, NaScratch *__restrict__ S) {
    grid_trigger();
    const int searchers = sh.hot ? sh.d : 0;
    if ((int)blockIdx.x >= searchers) {
        const int64_t total = sh.rows * sh.R, step = (int64_t)(gridDim.x - searchers) * kNaThreads;
        const int64_t first = (int64_t)(blockIdx.x - searchers) * kNaThreads + threadIdx.x;
        if ((reinterpret_cast<uintptr_t>(G) & 15) == 0) {
            for (int64_t e = first; e < (total >> 2); e += step)
                reinterpret_cast<float4 *>(G)[e] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            if (first < (total & 3)) G[(total & ~(int64_t)3) + first] = 0.0f;
        } else {
            for (int64_t e = first; e < total; e += step) G[e] = 0.0f;
        }
        return;
    }
    const int k = blockIdx.x;
    __shared__ int key[kNaTable];
    __shared__ unsigned count[kNaTable];
    __shared__ int over[8], slots;
    for (int i = threadIdx.x; i < kNaTable; i += kNaThreads) {
        key[i] = -1;
        count[i] = 0;
    }
    if (threadIdx.x < 8) over[threadIdx.x] = 0;
    if (threadIdx.x == 0) slots = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < kNaProbe; i += kNaThreads) {
        const int r = __ldg(idx + (n * i / kNaProbe) * sh.d + k);
        if (r < 0 || r >= sh.dims[k]) continue;
        unsigned h = ((unsigned)r * 2654435769u) >> 20;
        for (int probe = 0; probe < 32; ++probe, h = (h + 1) & (kNaTable - 1)) {  // at most half full
            const int was = atomicCAS(&key[h], -1, r);
            if (was == -1 || was == r) {
                atomicAdd(&count[h], 1u);
                break;
            }
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kNaTable; i += kNaThreads)
        for (int t = 0; t < 8; ++t)
            if (count[i] >= (8u << t)) atomicAdd(&over[t], 1);
    __syncthreads();
    int t = 0;
    while (t < 7 && over[t] && !gcpna::replicas(over[t], sh.R, sh.d)) ++t;
    const int word = gcpna::hot_word(over[t], sh.R, sh.d);
    if (word)
        for (int i = threadIdx.x; i < kNaTable; i += kNaThreads)
            if (count[i] >= (8u << t)) S->hot[k].row[atomicAdd(&slots, 1)] = key[i];
    if (threadIdx.x == 0) S->hot[k].word = word;
    const int floats = gcpna::hot_count(word) * gcpna::hot_replicas(word) * gcpna::row_floats(sh.R);
    for (int i = threadIdx.x; i < floats; i += kNaThreads) S->rep[k * gcpna::mode_floats(sh.d) + i] = 0.0f;
}

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

// Sampled gradient of a sample list.  A warp takes tiles of up to 32 consecutive
// samples: lane l reads sample l's coordinates, value and weight (the next
// tile's are in flight while this one is evaluated), then groups of L lanes
// take the tile's samples in turn, their row offsets, values and weights
// handed over by shuffles.  Lane g of a group owns columns V (g + L q) ..
// V (g + L q) + V - 1 for q < NQ; those past the rank are skipped, so rows
// need no padding.  Each lane keeps its own sample's loss and adds it in
// FP64 once per tile (three FP64 instructions per 32 samples).
// Reductions of a hot row go to one of its replicas (chosen by warp), folded
// afterwards; a lane looks its sample's rows up in a small table in shared
// memory.
// Bound by the row traffic through L2 (d rows gathered, d rows reduced per
// sample).  2^18 samples of the 2000 x 1500 x 1000 x 200 Zipf tensor at rank 32,
// drawn with gcp_sample and passed here: 99 to 105 us a pass, this kernel 42;
// 156 us with every reduction added to G itself (the ones that meet in one row
// are applied one after another, about 4.7 ns each); 745 us with one warp per
// sample walking 256 samples one after another on 128 blocks.
template <int D, int V, int NQ>
__global__ void __launch_bounds__(kNaThreads, (D <= 4 ? 3 : 2))
    k_na_grad(const NaShape sh, int loss, int64_t n, const int32_t *__restrict__ idx, const float *__restrict__ x,
              const float *__restrict__ w, const float *__restrict__ A, float *__restrict__ G,
              NaScratch *__restrict__ S) {
    constexpr int C = V * NQ;  // columns per lane
    constexpr int kBuckets = 64;
    __shared__ int s_row[D][kBuckets];             // -1: empty
    __shared__ unsigned char s_slot[D][kBuckets];
    __shared__ int s_hot[D];                       // hot_word
    grid_wait();  // G is cleared and the hot rows are known
    grid_trigger();
    if (sh.hot) {
        if (threadIdx.x < D) s_hot[threadIdx.x] = gcpna::hot_word_for(S->hot[threadIdx.x].word, sh.R, D);
        for (int i = threadIdx.x; i < D * kBuckets; i += kNaThreads) (&s_row[0][0])[i] = -1;
        __syncthreads();
        for (int i = threadIdx.x; i < D * gcpna::kHot; i += kNaThreads) {
            const int k = i / gcpna::kHot, j = i % gcpna::kHot;
            if (j >= gcpna::hot_count(s_hot[k])) continue;
            const int r = S->hot[k].row[j];
            unsigned h = ((unsigned)r * 2654435769u) >> 26;
            while (atomicCAS(&s_row[k][h], -1, r) != -1) h = (h + 1) & (kBuckets - 1);  // at most half full
            s_slot[k][h] = (unsigned char)j;
        }
        __syncthreads();
    }
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
    const int TS = sh.tile;
    const int64_t ntiles = (n + TS - 1) / TS;
    const int64_t nwarps = (int64_t)gridDim.x * kNaWarps;
    const int rf = gcpna::row_floats(sh.R);
    int rep[D];  // where this warp's replicas of a mode's hot rows start
#pragma unroll
    for (int k = 0; k < D; ++k) {
        rep[k] = k * gcpna::mode_floats(D);
        if (sh.hot && s_hot[k])
            rep[k] += (((int)blockIdx.x * kNaWarps + warp) & (gcpna::hot_replicas(s_hot[k]) - 1)) *
                      gcpna::hot_count(s_hot[k]) * rf;
    }
    int32_t ni[D];  // the next tile's sample of this lane
    float nx = 0.0f, nw = 0.0f;
    auto fetch = [&](int64_t tile) {
        const int64_t s = tile * TS + lane;
        if (lane < TS && s < n) {
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
        const bool in = lane < TS && tile * TS + lane < n;
        skipped += in && !ok;  // out-of-range coordinates: the sample is skipped and counted
        const unsigned okmask = __ballot_sync(0xFFFFFFFFu, in && ok);
        unsigned hot[(D + 3) / 4];  // per mode a byte: the row's hot slot, or 255
#pragma unroll
        for (int k = 0; k < D; ++k) {
            unsigned slot = 255u;
            if (sh.hot)
                for (unsigned h = ((unsigned)ni[k] * 2654435769u) >> 26;; h = (h + 1) & (kBuckets - 1)) {
                    const int r = s_row[k][h];  // an empty bucket ends the search
                    if (r == ni[k]) slot = s_slot[k][h];
                    if (r == ni[k] || r == -1) break;
                }
            hot[k / 4] = (k % 4 ? hot[k / 4] : 0u) | slot << (8 * (k % 4));
        }
        fetch(tile + nwarps);
        float myf = 0.0f;
        for (int it = 0; it * ngrp < TS; ++it) {
            const int src = it * ngrp + grp;
            const bool live = (okmask >> src) & 1u;  // uniform within the group
            const float xs = __shfl_sync(0xFFFFFFFFu, myx, src), ws = __shfl_sync(0xFFFFFFFFu, myw, src);
            int64_t off[D];
            unsigned hs[(D + 3) / 4];
#pragma unroll
            for (int i = 0; i < (D + 3) / 4; ++i) hs[i] = __shfl_sync(0xFFFFFFFFu, hot[i], src);
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
                const int slot = (int)((hs[k / 4] >> (8 * (k % 4))) & 255u);
                float *const g = slot == 255 ? G + off[k] : S->rep + rep[k] + slot * rf;
#pragma unroll
                for (int q = 0; q < NQ; ++q) {
                    if (!on[q]) continue;
                    float c[V];
#pragma unroll
                    for (int v = 0; v < V; ++v) c[v] = pre[V * q + v] * suf[k][V * q + v];
                    na_add<V>(g + col[q], c);
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
        S->partials[blockIdx.x] = t;
    }
}

// The last block: fixed-order sum of the block partials, loss_out[0] = loss,
// loss_out[1] = samples skipped for out-of-range coordinates.  The others, one
// per mode and hot row: the row's replicas added to G.
__global__ void __launch_bounds__(kNaThreads) k_na_finish(const NaShape sh, float *__restrict__ G, NaScratch *S,
                                                         int nblocks, double *loss_out) {
    grid_wait();
    if (blockIdx.x < gridDim.x - 1) {
        const int k = blockIdx.x / gcpna::kHot, j = blockIdx.x % gcpna::kHot;
        const int word = gcpna::hot_word_for(*const_cast<const volatile int *>(&S->hot[k].word), sh.R, sh.d);
        const int row = *const_cast<const volatile int *>(&S->hot[k].row[j]);  // both read once, then checked
        const int hot = gcpna::hot_count(word), nrep = gcpna::hot_replicas(word), rf = gcpna::row_floats(sh.R);
        const int c = threadIdx.x;
        if (j >= hot || c >= sh.R || !gcpna::row_in_mode(row, sh.dims[k])) return;
        const float *p = S->rep + k * gcpna::mode_floats(sh.d) + j * rf + c;
        float t = 0.0f;
        for (int r = 0; r < nrep; r += 4) {  // 4, 8, 16 or 32
            float v[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = p[(r + u) * hot * rf];
            t += (v[0] + v[1]) + (v[2] + v[3]);
        }
        G[(sh.rowoff[k] + row) * sh.R + c] += t;
        return;
    }
    __shared__ double2 red[kNaThreads];
    double2 t = make_double2(0.0, 0.0);
    for (int b = threadIdx.x; b < nblocks; b += kNaThreads) {
        t.x += S->partials[b].x;
        t.y += S->partials[b].y;
    }
    red[threadIdx.x] = t;
    __syncthreads();
    for (int h = kNaThreads / 2; h > 0; h >>= 1) {
        if (threadIdx.x < h) {
            red[threadIdx.x].x += red[threadIdx.x + h].x;
            red[threadIdx.x].y += red[threadIdx.x + h].y;
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        loss_out[0] = red[0].x;
        loss_out[1] = red[0].y;
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
                          NaScratch *);

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

// Device address of g_na_scratch, looked up once per device.  In host
// code the array's name is only a host-side stand-in, so the kernel must be
// given the address that cudaGetSymbolAddress returns for the current
// device.
std::mutex g_na_mutex;
NaScratch *g_na_addr[kNaMaxDevices] = {nullptr};

cudaError_t scratch_for_current_device(NaScratch **out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kNaMaxDevices) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lock(g_na_mutex);
    if (!g_na_addr[dev]) {
        void *p = nullptr;
        e = cudaGetSymbolAddress(&p, g_na_scratch);
        if (e != cudaSuccess) return e;
        g_na_addr[dev] = static_cast<NaScratch *>(p);
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
    NaScratch *scratch = nullptr;
    cudaError_t e = scratch_for_current_device(&scratch);
    if (e != cudaSuccess) return na_fail(GCP_ERR_CUDA, cudaGetErrorString(e));
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    // A hot row needs that many reductions in one line to matter: 2^14
    // samples of which a fifth meet in one row are 15 us, less than two
    // launches; from there on the list is searched.
    sh.d = ndim;
    sh.rows = rows;
    sh.hot = nsamples >= 1 << 14;
    const int64_t clear = (rows * rank / 4 + kNaThreads - 1) / kNaThreads;
    k_na_setup<<<(sh.hot ? ndim : 0) + (int)std::max<int64_t>(1, std::min<int64_t>(clear, 1216)), kNaThreads, 0, st>>>(
        sh, nsamples, idx, G, scratch);
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
        const int most = std::min(std::max(1, per_sm) * sms, kNaMaxBlocks);
        sh.tile = gcpk::fused_tile(nsamples, plan.log2L, most);
        const int64_t ntiles = (nsamples + sh.tile - 1) / sh.tile;
        nblocks = (int)std::min<int64_t>((ntiles + kNaWarps - 1) / kNaWarps, most);
        e = gcpk::launch_dependent(k, nblocks, kNaThreads, 0, st, sh, loss, nsamples, idx, x, w, A, G, scratch);
        if (e != cudaSuccess) return na_fail(GCP_ERR_CUDA, cudaGetErrorString(e));
    }
    e = gcpk::launch_dependent(k_na_finish, (sh.hot ? ndim * gcpna::kHot : 0) + 1, kNaThreads, 0, st, sh, G, scratch, nblocks,
                               loss_out);
    if (e != cudaSuccess) return na_fail(GCP_ERR_CUDA, cudaGetErrorString(e));
    if ((e = cudaGetLastError()) != cudaSuccess) return na_fail(GCP_ERR_CUDA, cudaGetErrorString(e));
    return GCP_OK;
}
