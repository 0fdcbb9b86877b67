// gcp_api.cu -- the C ABI of include/gcp.h: context set-up, argument checks,
// the stratified weights of Sec. 3.1.1, kernel launches and the GCP-Adam
// epoch loop (Algorithm 2 on one GPU).
#include <cuda_bf16.h>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <algorithm>
#include <new>
#include <string>
#include <vector>

#include "gcp_device.cuh"
#include "gcp_internal.h"

namespace {

thread_local std::string g_create_err;

struct DeviceGuard {  // make the context's device current for one call
    int prev = -1;
    explicit DeviceGuard(int dev) {
        cudaGetDevice(&prev);
        if (prev != dev) cudaSetDevice(dev);
    }
    ~DeviceGuard() {
        int cur = -1;
        cudaGetDevice(&cur);
        if (prev >= 0 && cur != prev) cudaSetDevice(prev);
    }
};

gcp_status fail(gcp_ctx *c, gcp_status code, const std::string &msg) {
    if (c)
        c->err = msg;
    else
        g_create_err = msg;
    return code;
}

gcp_status cuda_fail(gcp_ctx *c, cudaError_t e, const char *what) {
    return fail(c, e == cudaErrorMemoryAllocation ? GCP_ERR_OOM : GCP_ERR_CUDA,
                std::string(what) + ": " + cudaGetErrorString(e));
}

#define GCP_CUDA(ctx, call)                                      \
    do {                                                         \
        cudaError_t e_ = (call);                                 \
        if (e_ != cudaSuccess) return cuda_fail(ctx, e_, #call); \
    } while (0)

constexpr int64_t kStageBytes = 8 << 20;  // rows_out, rows_in

uint64_t next_pow2(uint64_t v) {
    uint64_t p = 1;
    while (p < v) p <<= 1;
    return p;
}

// status word -> first gcp_status code set
gcp_status status_code(int bits) {
    for (int c = 1; c < 31; ++c)
        if (bits & (1 << c)) return (gcp_status)c;
    return GCP_OK;
}

const char *status_text(gcp_status s) {
    switch (s) {
    case GCP_ERR_DUPLICATE: return "duplicate nonzero coordinates";
    case GCP_ERR_HASH_FULL: return "nonzero hash set is full";
    case GCP_ERR_SAMPLER_EXHAUSTED: return "a zero draw hit nonzeros max_attempts times (tensor too dense)";
    case GCP_ERR_NONFINITE: return "non-finite loss";
    case GCP_ERR_ARG: return "non-finite value in the dense tensor";
    case GCP_ERR_DOMAIN: return "value outside the loss's domain";
    default: return "device error";
    }
}

// Read and clear the device status word; synchronises the stream.
gcp_status collect(gcp_ctx *c) {
    GCP_CUDA(c, cudaMemcpyAsync(c->h_status, c->status, sizeof(int), cudaMemcpyDeviceToHost, c->st));
    GCP_CUDA(c, cudaStreamSynchronize(c->st));
    const int bits = *c->h_status;
    if (bits) {
        GCP_CUDA(c, cudaMemsetAsync(c->status, 0, sizeof(int), c->st));
        const gcp_status s = status_code(bits);
        return fail(c, s, status_text(s));
    }
    return GCP_OK;
}

void destroy_buffers(gcp_ctx *c) {
    cudaFree(c->rec);
    cudaFree(c->hkeys);
    cudaFree(c->X);
    cudaFree(c->A);
    cudaFree(c->stage);
    cudaFree(c->Abf);
    cudaFree(c->G);
    cudaFree(c->B);
    cudaFree(c->C);
    cudaFree(c->partials);
    cudaFree(c->dloss);
    cudaFree(c->status);
    cudaFree(c->det_scratch);
    if (c->det_side) cudaStreamDestroy(c->det_side);
    if (c->det_fork) cudaEventDestroy(c->det_fork);
    if (c->det_join) cudaEventDestroy(c->det_join);
    cudaFree(c->nf_coord);
    cudaFree(c->nf_val);
    cudaFree(c->hot_slot);
    cudaFree(c->hot_row);
    cudaFree(c->Grep);
    cudaFree(c->bk_A);
    cudaFree(c->bk_B);
    cudaFree(c->bk_C);
    cudaFreeHost(c->h_status);
    cudaFreeHost(c->h_loss);
    for (auto &ev : c->prof_ev) {
        cudaEventDestroy(ev.first);
        cudaEventDestroy(ev.second);
    }
    c->prof_ev.clear();
}

// Event pair for the next timed launch (reused across reads).
gcp_status prof_begin(gcp_ctx *c, cudaEvent_t *stop) {
    *stop = nullptr;
    if (!c->prof) return GCP_OK;
    if (c->prof_used == c->prof_ev.size()) {
        std::pair<cudaEvent_t, cudaEvent_t> ev;
        GCP_CUDA(c, cudaEventCreate(&ev.first));
        GCP_CUDA(c, cudaEventCreate(&ev.second));
        c->prof_ev.push_back(ev);
    }
    auto &ev = c->prof_ev[c->prof_used++];
    GCP_CUDA(c, cudaEventRecord(ev.first, c->st));
    *stop = ev.second;
    return GCP_OK;
}

// Shape, options and model buffers common to sparse and dense contexts.
gcp_status init_common(gcp_ctx *c, int32_t ndim, const int64_t *dims, int32_t rank, int32_t loss,
                       const gcp_options *opt) {
    if (ndim < 2 || ndim > GCP_MAX_NDIM) return fail(nullptr, GCP_ERR_ARG, "ndim must be in 2..8");
    if (!dims) return fail(nullptr, GCP_ERR_ARG, "dims is NULL");
    if (rank < 1 || rank > GCP_MAX_RANK) return fail(nullptr, GCP_ERR_ARG, "rank must be in 1..128");
    if (loss < GCP_GAUSSIAN || loss > GCP_GAMMA) return fail(nullptr, GCP_ERR_ARG, "unknown loss");
    gcp_options_default(&c->opt);
    if (opt) c->opt = *opt;
    if (c->opt.factor_dtype != GCP_FP32 && c->opt.factor_dtype != GCP_BF16)
        return fail(nullptr, GCP_ERR_ARG, "unknown factor dtype");
    if (c->opt.mttkrp != GCP_MTTKRP_ATOMIC && c->opt.mttkrp != GCP_MTTKRP_DETERMINISTIC &&
        c->opt.mttkrp != GCP_MTTKRP_NONFUSED)
        return fail(nullptr, GCP_ERR_ARG, "unknown MTTKRP variant");
    if (c->opt.max_attempts < 0) return fail(nullptr, GCP_ERR_ARG, "max_attempts < 0");
    if (c->opt.max_attempts == 0) c->opt.max_attempts = 64;
    if (c->opt.hash_max_load == 0.0) c->opt.hash_max_load = 0.3;
    if (!(c->opt.hash_max_load > 0.0 && c->opt.hash_max_load <= 0.5))
        return fail(nullptr, GCP_ERR_ARG, "hash_max_load must be in (0, 0.5]");
    c->d = ndim;
    c->R = rank;
    c->loss = loss;
    c->st = static_cast<cudaStream_t>(c->opt.stream);
    cudaGetDevice(&c->device);
    unsigned __int128 M = 1;
    for (int k = 0; k < ndim; ++k) {
        if (dims[k] < 1 || dims[k] > INT32_MAX) return fail(nullptr, GCP_ERR_ARG, "mode size out of range");
        c->dims[k] = dims[k];
        M *= (unsigned __int128)dims[k];
        if (M >= ((unsigned __int128)1 << 63)) return fail(nullptr, GCP_ERR_ARG, "prod(dims) must be < 2^63");
    }
    c->M = (double)(uint64_t)M;
    c->stride[ndim - 1] = 1;
    for (int k = ndim - 2; k >= 0; --k) c->stride[k] = c->stride[k + 1] * (uint64_t)dims[k + 1];
    c->total_rows = 0;
    for (int k = 0; k < ndim; ++k) {
        c->rowoff[k] = c->total_rows;
        c->total_rows += dims[k];
    }
    // Row length padded to 4 x a power of two, and the columns of it that a
    // lane owns.  Eight halve the work that each group of lanes repeats
    // (index arithmetic, loss, shuffles); four let a group's reduction cover
    // a whole row of up to 128 bytes with one instruction and leave registers
    // for a fourth block per SM.  A pass without reductions takes eight
    // wherever there are eight columns, and still fits four blocks (2^19
    // samples of the 4-way Zipf tensor, rank 32 BF16: kernel 42.8 -> 35.8 us).
    // A gradient pass takes eight from rank 33 on (2^20 samples of 2 to 8
    // modes at ranks 33 to 65: 12 to 27% faster).  At a padded rank of 32 it
    // takes eight for two modes (ranks 17 to 28, 2^16 and 2^20 samples: 4 to 22%
    // faster, rank 32 12%), and for three and four where one lane's second quad
    // is in use at most: ranks 17 to 20 are five quads of columns (1 to 13%
    // faster, all four ranks alike), ranks 21 to 24 six (2^20 samples 6 to 8%
    // slower, 2^16 between 4% slower and 3% faster), 26 and 28 slower by up to
    // 19%.  With five modes and six it costs registers (ranks 17 to 20: five
    // modes 1 to 16% slower, six between 13% slower and 9% faster).
    int Rp = 4;
    while (Rp < rank) Rp <<= 1;
    c->Rp = Rp;
    c->cols = Rp >= 64 || (Rp == 32 && (ndim == 2 || (rank <= 20 && ndim <= 4))) ? 8 : 4;
    c->eval_cols = Rp >= 8 ? 8 : 4;
    if (c->opt.lane_cols == 4 || (c->opt.lane_cols == 8 && Rp >= 8)) c->cols = c->eval_cols = c->opt.lane_cols;
    else if (c->opt.lane_cols != 0) return fail(nullptr, GCP_ERR_ARG, "lane_cols must be 0, 4 or 8");
    while ((c->cols << c->log2L) < Rp) ++c->log2L;
    while ((c->eval_cols << c->eval_log2L) < Rp) ++c->eval_log2L;
    if ((double)c->total_rows * c->Rp >= 2147483647.0)
        return fail(nullptr, GCP_ERR_ARG, "sum of mode sizes x padded rank must be < 2^31");

    const size_t nparam = (size_t)c->total_rows * c->Rp;
    cudaError_t e;
    if ((e = cudaMalloc(&c->A, nparam * 4)) || (e = cudaMalloc(&c->G, nparam * 4)) ||
        (e = cudaMalloc(&c->B, nparam * 4)) || (e = cudaMalloc(&c->C, nparam * 4)) ||
        (e = cudaMalloc(&c->dloss, 4 * sizeof(double))) || (e = cudaMalloc(&c->status, sizeof(int))) ||
        (e = cudaMallocHost(&c->h_status, sizeof(int))) || (e = cudaMallocHost(&c->h_loss, 4 * sizeof(double))))
        return cuda_fail(nullptr, e, "allocating model buffers");
    if (c->R != c->Rp) {
        c->stage_rows = std::min<int64_t>(c->total_rows, std::max<int64_t>(1, kStageBytes / (4 * c->R)));
        if ((e = cudaMalloc(&c->stage, (size_t)c->stage_rows * c->R * 4)))
            return cuda_fail(nullptr, e, "allocating the staging rows");
    }
    if (c->opt.factor_dtype == GCP_BF16 && (e = cudaMalloc(&c->Abf, nparam * 2)))
        return cuda_fail(nullptr, e, "allocating BF16 factors");
    c->max_blocks = gcpk::fused_max_blocks(ndim, c->opt.factor_dtype == GCP_BF16, c->cols);
    if ((e = cudaMalloc(&c->partials, (size_t)c->max_blocks * 4 * sizeof(double))))
        return cuda_fail(nullptr, e, "allocating partials");
    if ((e = cudaMemsetAsync(c->A, 0, nparam * 4, c->st)) || (e = cudaMemsetAsync(c->G, 0, nparam * 4, c->st)) ||
        (e = cudaMemsetAsync(c->B, 0, nparam * 4, c->st)) || (e = cudaMemsetAsync(c->C, 0, nparam * 4, c->st)) ||
        (e = cudaMemsetAsync(c->status, 0, sizeof(int), c->st)) ||
        (c->Abf && (e = cudaMemsetAsync(c->Abf, 0, nparam * 2, c->st))))
        return cuda_fail(nullptr, e, "clearing model buffers");
    return GCP_OK;
}

gcpk::SampleSpec sample_spec(const gcp_ctx *c, uint64_t iter, int64_t p, int64_t q) {
    gcpk::SampleSpec s{};
    s.d = c->d;
    for (int k = 0; k < c->d; ++k) {
        s.dims[k] = c->dims[k];
        s.stride[k] = c->stride[k];
    }
    s.nnz = c->nnz;
    s.rec = c->rec;
    s.rec_words = c->rec_words;
    s.hkeys = c->hkeys;
    s.hbmask = c->hbmask;
    s.dense = c->X;
    s.seed = c->opt.seed;
    s.iter = iter;
    s.p = p;
    s.q = q;
    s.sampling = c->opt.sampling;
    s.max_attempts = c->opt.max_attempts;
    s.status = c->status;
    return s;
}

// Per-sample weights of Sec. 3.1.1: N/p for nonzeros, (M-N)/q for zeros;
// semi-stratified zero candidates cover all M cells (M/q); dense uniform
// sampling weighs each of the p cells M/p.
void weights(const gcp_ctx *c, int64_t p, int64_t q, double &w_nz, double &w_z) {
    if (c->opt.sampling == GCP_SAMPLING_UNIFORM) {
        w_nz = p > 0 ? c->M / (double)p : 0.0;
        w_z = 0.0;
        return;
    }
    w_nz = p > 0 ? (double)c->nnz / (double)p : 0.0;
    if (c->opt.sampling == GCP_SAMPLING_SEMI_STRATIFIED)
        w_z = q > 0 ? c->M / (double)q : 0.0;
    else
        w_z = q > 0 ? (c->M - (double)c->nnz) / (double)q : 0.0;
}

gcp_status check_counts(gcp_ctx *c, int64_t p, int64_t q) {
    if (p < 0 || q < 0) return fail(c, GCP_ERR_ARG, "negative sample count");
    if (c->dense && q != 0) return fail(c, GCP_ERR_ARG, "dense tensors take p uniform samples and q = 0");
    if (p + q >= ((int64_t)1 << 31)) return fail(c, GCP_ERR_ARG, "p + q must be below 2^31 per call");
    return GCP_OK;
}

// Whether a hot row's replicas lie one after another, instead of in planes of
// all hot rows.  Where single rows take far more of the nonzeros than a uniform
// tensor's, the reductions gather in few lines, and it counts how those fall on
// the L2 slices.  Rows of two lines and more (padded rank 64 and 128) do better
// one after another: training steps of 2^20 and 2^19 samples on eight Zipf
// tensors of 3 and 4 modes 0 to 5% faster than in planes, none slower by more
// than 0.5% (2000 x 1500 x 1000 x 200 at rank 64 207 -> 193 us).  Shorter rows
// do not: at ranks 4 to 32, each replica in a line of its own, from 9% faster
// (4000 x 3000 x 2000 x 500 at rank 32 244 -> 222 us) to 12% slower (1000^4 216
// -> 238 us at rank 32, 103 -> 115 at rank 4), on average slower.  Without skew
// planes, compact per warp, are the better layout, and above order 4, where a
// row's stride other than Rp costs registers (dense 5-way gradient 326 against
// 334 us), they are kept always.
bool replica_lines(const gcp_ctx *c) { return c->d <= 4 && c->Rp >= 64 && c->share_nz > 2.0 * c->share_cell; }

// Replicas of the hot rows for a sample set.  Two things ask for them:
//  - time: the reductions that meet in one 128-byte line are applied one after
//    another, about 4.7 ns each (with no replicas a step of 2^21 samples of
//    the 4-way Zipf tensor takes 0.78 ms and the dense 5-way gradient of 2^22
//    samples 1.96 ms: their hottest line's expected count x 4.2-4.7 ns), so the
//    hottest line bounds the pass from below by that count x 4.7 ns / nrep.  A
//    line holds 32 / Rp rows of a padded rank below 32.  This chain is to be
//    under 6% of the pass's row traffic (2 x 4 B x D Rp per sample at about 9
//    TB/s) or under 4 us, less than the latency of the shortest pass;
//  - precision: the terms of a row are added in FP32 one after another within
//    a replica, so the hottest row's expected terms are to be at most 32 in
//    each.  With 64 replicas whatever the count, rows of up to about 2,000
//    terms had that too, and shorter chains gain nothing against the FP64
//    gradient, relative 2-norm: 2,000 samples on modes of 30 to 50 rows (66
//    terms a row) 8.3e-8 with no replicas, 4.9e-8, 4.5e-8 and 4.5e-8 with 4, 16
//    and 64; 2^16 samples on modes of 172 to 25,000 rows (381 terms) 2.7e-7,
//    8.2e-8, 4.8e-8 and 4.5e-8.
// Against them, every replica costs the fold 8 B per entry of every hot row.
// The count is rounded up to one the folds are built for, and 64 is the most:
// rows with more than 2,048 terms have longer chains (the two shapes below
// with 64 about 5,000 and 3,300 terms a replica at most), and so have rows
// without replicas, in modes of more than 512 rows.
// Measured with 0 / 4 / 16 / 64 replicas: step of the 4-way Zipf tensor, rank
// 32, 2^21 samples 784 / 461 / 276 / 222 us (rule: 64); dense 5-way gradient,
// rank 16, 2^22 samples 1956 / 724 / 402 / 325 us (64); 172 x 25,000 x 300,
// rank 50, 2^16 samples 21.6 / 20.3 / 20.9 / 27.1 us (16); 211 x 187 x 95 x 24
// Zipf, rank 10, 10^4 samples 11.9 / 8.8 / 8.8 / 9.0 us per fit iteration (64);
// 8 local steps of 16 clients, 500 hot rows and 16,384 samples each, 265 / 268
// / 296 / 457 us (4).
int replicas_for(const gcp_ctx *c, int64_t p, int64_t q) {
    if (!c->Grep) return 0;
    const double line = c->Rp >= 32 ? 1.0 : 32.0 / c->Rp;  // rows of a 128-byte line
    const double cell = std::min(1.0, c->share_cell * line);
    const bool uniform = c->opt.sampling == GCP_SAMPLING_UNIFORM;
    const double hits = uniform ? (double)p * cell : (double)p * c->share_nz + (double)q * cell;
    const double terms = uniform ? (double)p * c->share_cell
                                 : (double)p * c->share_nz + (double)q * c->share_cell;
    const double pass = (double)(p + q) * 8.0 * c->d * c->Rp / 9000.0;  // ns
    const double want = std::max(hits * 4.7 / std::max(0.06 * pass, 4000.0), terms / 32.0);
    return want <= 1.0 ? 0 : (want <= 4.0 ? 4 : (want <= 16.0 ? 16 : gcpk::kReplicas));
}

// One fused pass: loss always, gradient into c->G when `grad`.
}  // namespace

// The fused-pass parameters of one sample set of a context (also used for
// each client of a batch).
gcpk::FusedSpec gcpk_make_spec(const gcp_ctx *c, uint64_t iter, int64_t p, int64_t q, bool grad,
                               const float *dscale, double *w_nz_out, double *w_z_out) {
    double w_nz, w_z;
    weights(c, p, q, w_nz, w_z);
    gcpk::FusedSpec f{};
    f.s = sample_spec(c, iter, p, q);
    f.F = c->Abf ? c->Abf : (const void *)c->A;
    f.G = grad ? c->G : nullptr;
    f.Rp = c->Rp;
    f.R = c->R;
    f.log2L = grad ? c->log2L : c->eval_log2L;
    f.tile = gcpk::fused_tile(p + q, c->log2L, c->max_blocks);
    // Beside the end of the grid before, a pass draws its first samples.  For
    // small sample sets that and the launch itself are much of the call: a
    // step of 2,000 samples takes 6.5 us instead of 10.3, of 2^17 20.1 instead
    // of 22.6 (4999 x 3001 x 777, rank 20).  Large passes fill the GPU, and
    // blocks that arrive while the epilogue still runs cost more than they
    // gain: 2^20 samples at rank 32 on the Zipf tensor 128 against 121 us, a
    // step of the 121.6 M parameter model 1.3% slower.
    f.dependent = p + q <= (int64_t)1 << 19;
    for (int k = 0; k < c->d; ++k) f.rowoff[k] = (int)c->rowoff[k];
    f.loss = c->loss;
    f.w_nz = (float)w_nz;
    f.w_z = (float)w_z;
    f.dscale = dscale;
    f.partials = c->partials;
    f.nrep = grad ? replicas_for(c, p, q) : 0;
    for (int k = 0; k < c->d; ++k) f.small_base[k] = f.nrep ? c->small_base[k] : -1;
    f.Grep = f.nrep ? c->Grep : nullptr;
    f.Htot = f.nrep ? c->Htot : 0;
    f.rplane = replica_lines(c) ? c->Rp : c->Htot * c->Rp;
    f.rstride = replica_lines(c) ? f.nrep * c->Rp : c->Rp;
    if (w_nz_out) *w_nz_out = w_nz;
    if (w_z_out) *w_z_out = w_z;
    return f;
}

gcp_status gcpk_check_counts(gcp_ctx *c, int64_t p, int64_t q) { return check_counts(c, p, q); }

bool gcpk_begin_gradient(gcp_ctx *c) {
    cudaStreamCaptureStatus status = cudaStreamCaptureStatusNone;
    unsigned long long id = 0;
    bool known = true;
    if (cudaStreamGetCaptureInfo(c->st, &status, &id) != cudaSuccess) {
        cudaGetLastError();  // the legacy stream while another thread captures: not this call's error
        known = false;
    } else if (status == cudaStreamCaptureStatusNone) {
        id = 0;
    } else {
        c->g_captured = true;
    }
    const bool clear = known && c->g_clear && c->g_capture == id && (id != 0 || !c->g_captured);
    c->g_clear = false;
    c->g_capture = id;
    return clear;
}

namespace {

// Whether kernels of the context can write n bytes at p directly: device
// memory of its device or managed memory, aligned for `align`-byte accesses.
// Other pointers (host memory, another device) go through the copy calls,
// which say what is wrong with the ones they do not take.
bool kernel_writable(const gcp_ctx *c, const void *p, size_t align) {
    if (reinterpret_cast<uintptr_t>(p) % align) return false;
    cudaPointerAttributes at{};
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
        cudaGetLastError();  // not a sticky error
        return false;
    }
    return at.type == cudaMemoryTypeManaged || (at.type == cudaMemoryTypeDevice && at.device == c->device);
}

// Where the results of a fused pass go besides the context's own buffers.
struct Outputs {
    float *G = nullptr;       // unpadded gradient (host or device), or null
    double *dloss = nullptr;  // device loss, or null
    bool host = false;        // the pinned mirrors are read after a synchronisation
};

// The loss finish of a pass of `blocks` partials.  `copy_loss` tells whether
// the caller's device double still has to be copied (a pointer that the
// kernels cannot write).
gcpk::LossSpec loss_spec(gcp_ctx *c, int blocks, double w_nz, double w_z, const Outputs &o, bool *copy_loss) {
    gcpk::LossSpec l{};
    l.partials = c->partials;
    l.nblocks = blocks;
    l.w_nz = w_nz;
    l.w_z = w_z;
    l.dloss = c->dloss;
    l.status = c->status;
    const bool direct = o.dloss && kernel_writable(c, o.dloss, sizeof(double));
    l.out = direct ? o.dloss : nullptr;
    *copy_loss = o.dloss && !direct;
    if (o.host) {
        l.h_loss = c->h_loss;
        l.h_status = c->h_status;
    }
    return l;
}

gcp_status copy_loss_out(gcp_ctx *c, double *dloss_out) {
    GCP_CUDA(c, cudaMemcpyAsync(dloss_out, c->dloss, sizeof(double), cudaMemcpyDeviceToDevice, c->st));
    return GCP_OK;
}

// After a pass with Outputs::host: wait, then report the device errors that
// the loss finish mirrored (clearing them).
gcp_status host_result(gcp_ctx *c) {
    GCP_CUDA(c, cudaStreamSynchronize(c->st));
    const int bits = *c->h_status;
    if (!bits) return GCP_OK;
    GCP_CUDA(c, cudaMemsetAsync(c->status, 0, sizeof(int), c->st));
    const gcp_status s = status_code(bits);
    return fail(c, s, status_text(s));
}

gcp_status copy_grad_out(gcp_ctx *c, float *G_out);

gcp_status run_fused(gcp_ctx *c, uint64_t iter, int64_t p, int64_t q, bool grad, const float *dscale,
                     const Outputs &out) {
    gcp_status s = check_counts(c, p, q);
    if (s) return s;
    double w_nz, w_z;
    gcpk::FusedSpec f = gcpk_make_spec(c, iter, p, q, grad, dscale, &w_nz, &w_z);
    if (grad) {
        gcpk_begin_gradient(c);  // cleared whatever it returns: the pass starts beside this kernel
        GCP_CUDA(c, gcpk::launch_clear(c->G, c->total_rows * c->Rp, c->st));
    }
    int blocks = 0;
    cudaEvent_t stop = nullptr;
    if ((s = prof_begin(c, &stop))) return s;
    if (grad && c->opt.mttkrp == GCP_MTTKRP_DETERMINISTIC) {
        s = gcpk_det_grad(c, f, &blocks);
        if (s) return s;
    } else if (grad && c->opt.mttkrp == GCP_MTTKRP_NONFUSED) {
        const int64_t S = p + q;
        if (S > c->nf_cap) {  // grow the gradient-tensor buffers
            cudaFree(c->nf_coord);
            cudaFree(c->nf_val);
            c->nf_coord = nullptr;
            c->nf_val = nullptr;
            c->nf_cap = 0;
            GCP_CUDA(c, cudaMalloc(&c->nf_coord, (size_t)S * c->d * 4));
            GCP_CUDA(c, cudaMalloc(&c->nf_val, (size_t)S * 4));
            c->nf_cap = S;
        }
        gcpk::FusedSpec m = f;  // pass 1: sampling, model, loss; writes the gradient tensor
        m.G = nullptr;
        m.Ycoord = c->nf_coord;
        m.Yval = c->nf_val;
        m.ystride = c->d;
        m.vstride = 1;
        m.log2L = c->eval_log2L;
        GCP_CUDA(c, gcpk::launch_fused_eval(m, c->Abf != nullptr, c->eval_cols, c->max_blocks, c->st, &blocks));
        m.G = c->G;  // pass 2: MTTKRP of the stored gradient tensor
        m.log2L = c->log2L;
        GCP_CUDA(c, gcpk::launch_mttkrp_nonfused(m, f.nrep ? c->hot_slot : nullptr, c->Abf != nullptr, c->cols,
                                                 c->max_blocks, c->st));
    } else if (grad) {
        GCP_CUDA(c, gcpk::launch_fused(f, c->Abf != nullptr, c->cols, c->max_blocks, c->st, &blocks));
    } else {
        GCP_CUDA(c, gcpk::launch_fused_eval(f, c->Abf != nullptr, c->eval_cols, c->max_blocks, c->st, &blocks));
    }
    if (stop) GCP_CUDA(c, cudaEventRecord(stop, c->st));
    bool copy_loss = false;
    const gcpk::LossSpec loss = loss_spec(c, blocks, w_nz, w_z, out, &copy_loss);
    bool copy_grad = false;
    if (grad) {
        gcpk::GradOutSpec go{};
        go.loss = loss;
        go.rows = c->total_rows;
        go.Rp = c->Rp;
        go.R = c->R;
        go.G = c->G;
        if (c->opt.mttkrp != GCP_MTTKRP_DETERMINISTIC && f.nrep) {
            go.Htot = f.Htot;
            go.rstride = f.rstride;
            go.rplane = f.rplane;
            go.nrep = f.nrep;
            go.Grep = f.Grep;
            go.hot_slot = c->hot_slot;
            go.hot_row = c->hot_row;
        }
        const bool direct = out.G && kernel_writable(c, out.G, sizeof(float));
        go.out = direct ? out.G : nullptr;
        copy_grad = out.G && !direct;
        GCP_CUDA(c, gcpk::launch_grad_finish(go, c->st));
    } else {
        GCP_CUDA(c, gcpk::launch_finish_loss(loss, c->st));
    }
    if (copy_grad && (s = copy_grad_out(c, out.G))) return s;
    if (copy_loss && (s = copy_loss_out(c, out.dloss))) return s;
    return GCP_OK;
}

gcp_status adam_step_impl(gcp_ctx *c, const gcp_adam_params *prm, int64_t t) {
    if (t < 1) return fail(c, GCP_ERR_ARG, "Adam step t must be >= 1");
    if (!(prm->beta1 >= 0.0 && prm->beta1 < 1.0 && prm->beta2 >= 0.0 && prm->beta2 < 1.0 && prm->eps >= 0.0))
        return fail(c, GCP_ERR_ARG, "Adam parameters out of range");
    DeviceGuard g(c->device);
    const double c1 = 1.0 - std::pow(prm->beta1, (double)t), c2 = 1.0 - std::pow(prm->beta2, (double)t);
    GCP_CUDA(c, gcpk::launch_adam((int64_t)c->total_rows * c->Rp, c->Rp, c->R, c->A, c->B, c->C, c->G,
                                  (float)prm->lr, (float)prm->beta1, (float)prm->beta2, (float)(1.0 / c1),
                                  (float)(1.0 / c2), (float)prm->eps, (float)prm->lower, c->Abf, c->st));
    return GCP_OK;
}


// One training step: sampled gradient of iteration `iter` and Adam step t.
// With the atomic MTTKRP the epilogue (replica fold, loss finish, Adam, G
// cleared for the next step) is one launch after the fused pass.
// dloss_out (device, nullable) receives the loss.
gcp_status do_step(gcp_ctx *c, uint64_t iter, int64_t p, int64_t q, const gcp_adam_params *prm, int64_t t,
                   double *dloss_out) {
    gcp_status s;
    Outputs out;
    out.dloss = dloss_out;
    if (c->opt.mttkrp != GCP_MTTKRP_ATOMIC) {
        if ((s = run_fused(c, iter, p, q, true, nullptr, out))) return s;
        return adam_step_impl(c, prm, t);
    }
    if ((s = check_counts(c, p, q))) return s;
    double w_nz, w_z;
    gcpk::FusedSpec f = gcpk_make_spec(c, iter, p, q, true, nullptr, &w_nz, &w_z);
    if (!gcpk_begin_gradient(c)) GCP_CUDA(c, cudaMemsetAsync(c->G, 0, (size_t)c->total_rows * c->Rp * 4, c->st));
    int blocks = 0;
    cudaEvent_t stop = nullptr;
    if ((s = prof_begin(c, &stop))) return s;
    GCP_CUDA(c, gcpk::launch_fused(f, c->Abf != nullptr, c->cols, c->max_blocks, c->st, &blocks));
    if (stop) GCP_CUDA(c, cudaEventRecord(stop, c->st));
    const double c1 = 1.0 - std::pow(prm->beta1, (double)t), c2 = 1.0 - std::pow(prm->beta2, (double)t);
    gcpk::PostSpec ps{};
    ps.n = (int64_t)c->total_rows * c->Rp;
    ps.Rp = c->Rp;
    ps.R = c->R;
    ps.Htot = f.Htot;
    ps.rstride = f.rstride;
    ps.rplane = f.rplane;
    ps.nrep = f.nrep;
    ps.G = c->G;
    ps.Grep = f.Grep;
    ps.A = c->A;
    ps.B = c->B;
    ps.C = c->C;
    ps.Abf = c->Abf;
    ps.hot_slot = f.nrep ? c->hot_slot : nullptr;
    ps.hot_row = c->hot_row;
    ps.lr = (float)prm->lr;
    ps.beta1 = (float)prm->beta1;
    ps.beta2 = (float)prm->beta2;
    ps.c1inv = (float)(1.0 / c1);
    ps.c2inv = (float)(1.0 / c2);
    ps.eps = (float)prm->eps;
    ps.lower = (float)prm->lower;
    bool copy_loss = false;
    ps.loss = loss_spec(c, blocks, w_nz, w_z, out, &copy_loss);
    GCP_CUDA(c, gcpk::launch_post_step(ps, c->st));
    c->g_clear = true;
    return copy_loss ? copy_loss_out(c, dloss_out) : GCP_OK;
}

// Values of a dense tensor: bit GCP_ERR_ARG for a non-finite value, bit
// GCP_ERR_DOMAIN for one outside the loss's domain (the host checks of a
// sparse tensor's values, on the device).
__global__ void k_check_dense(const float *X, int64_t n, int loss, int *status) {
    int bad = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float x = X[i];
        if (!isfinite(x))
            bad |= 1 << GCP_ERR_ARG;
        else if ((loss == GCP_POISSON && x < 0.0f) || (loss == GCP_GAMMA && x <= 0.0f) ||
                 (loss == GCP_BERNOULLI_LOGIT && x != 1.0f && x != 0.0f))
            bad |= 1 << GCP_ERR_DOMAIN;
    }
    if (bad) atomicOr(status, bad);
}

// Factor matrices (src.A[k], I_k x R row-major, device memory) of the modes
// whose rows are row0 .. row0 + rows - 1 copied into the context's padded flat
// layout in one launch, one 16-byte quad of a padded row per thread; padding
// columns are written as zero and the BF16 copy, if any, is refreshed.  VEC:
// R and every pointer allow 16-byte loads.
struct FactorSrc {
    const float *A[GCP_MAX_NDIM];
    int64_t rowoff[GCP_MAX_NDIM + 1];  // first row of each mode, then the total
};

template <bool VEC>
__global__ void __launch_bounds__(256) k_stage_factors(FactorSrc src, int d, int R, int log2Rp, int64_t row0,
                                                       int64_t rows, float *A, __nv_bfloat16 *Abf) {
    gcpdev::grid_wait();  // the matrices and the context's factors may be in use by the grid before
    gcpdev::grid_trigger();
    const int log2Q = log2Rp - 2;
    const int64_t nq = rows << log2Q;
    for (int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x; e < nq; e += (int64_t)gridDim.x * 256) {
        const int64_t row = row0 + (e >> log2Q);
        const int col = (int)(e & ((1 << log2Q) - 1)) << 2;
        const float *base = src.A[0];
        int64_t first = 0;
#pragma unroll
        for (int k = 1; k < GCP_MAX_NDIM; ++k)  // constant indices only
            if (k < d && row >= src.rowoff[k]) {
                base = src.A[k];
                first = src.rowoff[k];
            }
        const float *a = base + (row - first) * R + col;
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (VEC) {
            if (col < R) v = *reinterpret_cast<const float4 *>(a);
        } else {
            if (col < R) v.x = a[0];
            if (col + 1 < R) v.y = a[1];
            if (col + 2 < R) v.z = a[2];
            if (col + 3 < R) v.w = a[3];
        }
        const int64_t q = (row << log2Q) + (col >> 2);
        reinterpret_cast<float4 *>(A)[q] = v;
        if (Abf) {
            const __nv_bfloat162 lo = __floats2bfloat162_rn(v.x, v.y), hi = __floats2bfloat162_rn(v.z, v.w);
            reinterpret_cast<uint2 *>(Abf)[q] = make_uint2(*reinterpret_cast<const unsigned *>(&lo),
                                                           *reinterpret_cast<const unsigned *>(&hi));
        }
    }
}

// y = s[0] * x elementwise (x and y may be the same array); s is FP64,
// rounded once to FP32.
__global__ void k_scale(const double *s, const float *x, float *y, int64_t n) {
    const float a = (float)__ldg(s);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        y[i] = a * x[i];
}

// Sum of squares of x[0..n) in FP64: block b adds its grid-stride elements
// in index order per thread, then a fixed tree; partial[b] holds the result.
__global__ void k_sumsq_blocks(const float *__restrict__ x, int64_t n, double *partial) {
    __shared__ double sh[256];
    double t = 0.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const double v = (double)x[i];
        t += v * v;
    }
    sh[threadIdx.x] = t;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) sh[threadIdx.x] += sh[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x == 0) partial[blockIdx.x] = sh[0];
}

// out[0] = sqrt(sum of the block partials), a fixed tree over one block; a
// non-finite result sets the status word.
__global__ void __launch_bounds__(256) k_sumsq_finish(const double *__restrict__ partial, int nblocks, double *out,
                                                      int *status) {
    __shared__ double sh[256];
    double t = 0.0;
    for (int b = threadIdx.x; b < nblocks; b += 256) t += partial[b];
    sh[threadIdx.x] = t;
    __syncthreads();
    for (int h = 128; h > 0; h >>= 1) {
        if ((int)threadIdx.x < h) sh[threadIdx.x] += sh[threadIdx.x + h];
        __syncthreads();
    }
    if (threadIdx.x != 0) return;
    out[0] = sqrt(sh[0]);
    if (!isfinite(sh[0])) atomicOr(status, 1 << GCP_ERR_NONFINITE);
}

// Rows row0 .. row0 + rows - 1 of padded device memory (row stride Rp) copied
// out to `out` (unpadded rows of R floats).  Device memory that kernels can
// write takes one kernel, except unpadded rows of 32 MB and more, where a
// plain copy is faster (486 MB: 164 against 174 us).  Host memory, and
// anything else, takes plain copies: of the rows as they are where there is
// no padding, else of unpadded rows staged kStageBytes at a time.  A strided
// copy moves each row by itself, about 2 ns a row out and 10 ns in: 10^6 rows
// of 10 floats 1.9 ms out and 10.5 ms in, against 0.29 ms staged; it stays for
// few rows, where it saves a launch (120 rows: 11 against 16 us out with the
// synchronisation, 3.4 against 9.2 us in).
constexpr int64_t kPlainBytes = 32 << 20, kStridedOut = 2048, kStridedIn = 512;

gcp_status rows_out(gcp_ctx *c, const float *src, int64_t row0, int64_t rows, float *out) {
    const float *p = src + row0 * c->Rp;
    const size_t row = (size_t)c->R * 4;
    if (!(c->R == c->Rp && rows * (int64_t)row >= kPlainBytes) && kernel_writable(c, out, sizeof(float))) {
        GCP_CUDA(c, gcpk::launch_unpad(p, c->Rp, c->R, rows, out, c->st));
        return GCP_OK;
    }
    if (c->R != c->Rp && rows <= kStridedOut) {
        GCP_CUDA(c, cudaMemcpy2DAsync(out, row, p, (size_t)c->Rp * 4, row, (size_t)rows, cudaMemcpyDefault, c->st));
        return GCP_OK;
    }
    if (c->R == c->Rp) {
        GCP_CUDA(c, cudaMemcpyAsync(out, p, row * rows, cudaMemcpyDefault, c->st));
        return GCP_OK;
    }
    for (int64_t r = 0; r < rows; r += c->stage_rows) {
        const int64_t n = std::min(c->stage_rows, rows - r);
        GCP_CUDA(c, gcpk::launch_unpad(p + r * c->Rp, c->Rp, c->R, n, c->stage, c->st));
        GCP_CUDA(c, cudaMemcpyAsync(reinterpret_cast<char *>(out) + r * row, c->stage, row * n, cudaMemcpyDefault,
                                    c->st));
    }
    return GCP_OK;
}

// Rows row0 .. row0 + rows - 1 of the factors (and of their BF16 copy) from
// the matrices src.A of the modes they span, device memory.
gcp_status stage_factors(gcp_ctx *c, const FactorSrc &src, int64_t row0, int64_t rows) {
    int log2Rp = 0;
    while ((1 << log2Rp) < c->Rp) ++log2Rp;
    bool vec = c->R % 4 == 0;
    for (int k = 0; k < c->d; ++k) vec = vec && (reinterpret_cast<uintptr_t>(src.A[k]) & 15) == 0;
    const int64_t want = (rows * (c->Rp / 4) + 255) / 256;
    const dim3 grid((unsigned)(want < 8192 ? want : 8192));
    auto *bf = static_cast<__nv_bfloat16 *>(c->Abf);
    if (vec)
        GCP_CUDA(c, gcpk::launch_dependent(k_stage_factors<true>, grid, 256, 0, c->st, src, c->d, c->R, log2Rp, row0,
                                           rows, c->A, bf));
    else
        GCP_CUDA(c, gcpk::launch_dependent(k_stage_factors<false>, grid, 256, 0, c->st, src, c->d, c->R, log2Rp, row0,
                                           rows, c->A, bf));
    return GCP_OK;
}

// The same from the unpadded rows at `in` (host or device): see rows_out.
gcp_status rows_in(gcp_ctx *c, int64_t row0, int64_t rows, const float *in) {
    FactorSrc src{};  // the modes' matrices as the kernel reads them, were all rows at `at`
    auto from = [&](const float *at, int64_t first) {
        for (int k = 0; k < c->d; ++k) {
            src.A[k] = at + (c->rowoff[k] - first) * c->R;
            src.rowoff[k] = c->rowoff[k];
        }
        src.rowoff[c->d] = c->total_rows;
    };
    const size_t row = (size_t)c->R * 4;
    const bool plain = c->R == c->Rp && !c->Abf && rows * (int64_t)row >= kPlainBytes;
    if (!plain && kernel_writable(c, in, sizeof(float))) {
        from(in, row0);
        return stage_factors(c, src, row0, rows);
    }
    if (c->R == c->Rp || rows <= kStridedIn) {
        if (c->R == c->Rp)
            GCP_CUDA(c, cudaMemcpyAsync(c->A + row0 * c->Rp, in, row * rows, cudaMemcpyDefault, c->st));
        else
            GCP_CUDA(c, cudaMemcpy2DAsync(c->A + row0 * c->Rp, (size_t)c->Rp * 4, in, row, row, (size_t)rows,
                                          cudaMemcpyDefault, c->st));
        if (c->Abf)
            GCP_CUDA(c, gcpk::launch_to_bf16(rows * c->Rp, c->A + row0 * c->Rp,
                                             static_cast<__nv_bfloat16 *>(c->Abf) + row0 * c->Rp, c->st));
        return GCP_OK;
    }
    for (int64_t r = 0; r < rows; r += c->stage_rows) {
        const int64_t n = std::min(c->stage_rows, rows - r);
        GCP_CUDA(c, cudaMemcpyAsync(c->stage, reinterpret_cast<const char *>(in) + r * row, row * n,
                                    cudaMemcpyDefault, c->st));
        from(c->stage, row0 + r);
        gcp_status s = stage_factors(c, src, row0 + r, n);
        if (s) return s;
    }
    return GCP_OK;
}

gcp_status copy_grad_out(gcp_ctx *c, float *G_out) { return rows_out(c, c->G, 0, c->total_rows, G_out); }

gcp_status refresh_bf16(gcp_ctx *c) {
    if (!c->Abf) return GCP_OK;
    GCP_CUDA(c, gcpk::launch_to_bf16((int64_t)c->total_rows * c->Rp, c->A, c->Abf, c->st));
    return GCP_OK;
}

// Rows that receive many gradient reductions per call get replicas: every
// row of a mode with at most 512 rows (each is hit by 1/I_k of the drawn
// cells), with contiguous slots so drawn cells find theirs by arithmetic;
// then, for larger modes, rows holding at least 1/512 of the nonzeros (hit
// by that share of the nonzero samples), at most 256 per mode, hottest
// first.  A nonzero record stores the slots of its rows.
gcp_status setup_hot_rows(gcp_ctx *c, const std::vector<int64_t> &counts) {
    std::vector<int> slot((size_t)c->total_rows, -1), row;
    for (int k = 0; k < c->d; ++k) c->share_cell = std::max(c->share_cell, 1.0 / (double)c->dims[k]);
    // nonzeros of the fullest row among those with replicas: the fullest of all
    // wherever there are any, since a mode of at most 512 rows has a row with
    // 1/512 of the nonzeros and a row without replicas holds less
    int64_t most = 0;
    for (int k = 0; k < c->d; ++k) {
        c->small_base[k] = -1;
        if (c->dims[k] > 512) continue;
        c->small_base[k] = (int)row.size();
        for (int64_t i = 0; i < c->dims[k]; ++i) {
            slot[(size_t)(c->rowoff[k] + i)] = (int)row.size();
            row.push_back((int)(c->rowoff[k] + i));
            if (!counts.empty()) most = std::max(most, counts[(size_t)(c->rowoff[k] + i)]);
        }
    }
    const int64_t floor_hot = (c->nnz + 511) / 512;  // the fewest nonzeros that are 1/512 of all
    for (int k = 0; k < c->d && !counts.empty(); ++k) {
        if (c->dims[k] <= 512) continue;
        std::vector<std::pair<int64_t, int>> hot;
        const int64_t *at = counts.data() + c->rowoff[k];
        for (int64_t i = 0; i < c->dims[k]; ++i)
            if (at[i] >= floor_hot) hot.push_back({at[i], (int)(c->rowoff[k] + i)});
        std::stable_sort(hot.begin(), hot.end(), [](const auto &x, const auto &y) { return x.first > y.first; });
        if (!hot.empty()) most = std::max(most, hot.front().first);
        if (hot.size() > 256) hot.resize(256);
        for (const auto &h : hot) {
            slot[(size_t)h.second] = (int)row.size();
            row.push_back(h.second);
        }
    }
    c->share_nz = counts.empty() ? 0.0 : (double)most / (double)c->nnz;
    c->Htot = (int)row.size();
    if (c->Htot == 0) return GCP_OK;
    const size_t rep_bytes = (size_t)gcpk::kReplicas * c->Htot * c->Rp * 4;
    cudaError_t e;
    if ((e = cudaMalloc(&c->hot_slot, slot.size() * 4)) || (e = cudaMalloc(&c->hot_row, row.size() * 4)) ||
        (e = cudaMalloc(&c->Grep, rep_bytes)) ||
        (e = cudaMemcpy(c->hot_slot, slot.data(), slot.size() * 4, cudaMemcpyHostToDevice)) ||
        (e = cudaMemcpy(c->hot_row, row.data(), row.size() * 4, cudaMemcpyHostToDevice)) ||
        (e = cudaMemsetAsync(c->Grep, 0, rep_bytes, c->st)))
        return cuda_fail(nullptr, e, "allocating hot-row replicas");
    return GCP_OK;
}

}  // namespace

void gcpk_set_noctx_error(const char *msg) { g_create_err = msg; }

// =================================================================== ABI
extern "C" {

void gcp_options_default(gcp_options *opt) {
    if (!opt) return;
    std::memset(opt, 0, sizeof(*opt));
    opt->factor_dtype = GCP_FP32;
    opt->mttkrp = GCP_MTTKRP_ATOMIC;
    opt->sampling = GCP_SAMPLING_STRATIFIED;
    opt->max_attempts = 64;
    opt->hash_max_load = 0.3;
}

gcp_status gcp_create(int32_t ndim, const int64_t *dims, int64_t nnz, const int32_t *coords, const float *vals,
                      int32_t rank, int32_t loss, const gcp_options *opt, gcp_ctx **out) {
    if (!out) return fail(nullptr, GCP_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (nnz < 1 || !coords || !vals) return fail(nullptr, GCP_ERR_ARG, "need nnz >= 1, coords and vals");
    if (opt && opt->sampling == GCP_SAMPLING_UNIFORM)
        return fail(nullptr, GCP_ERR_ARG, "uniform sampling is for dense tensors (gcp_create_dense)");
    // host checks of the nonzeros
    if (ndim >= 2 && ndim <= GCP_MAX_NDIM && dims) {
        for (int64_t e = 0; e < nnz; ++e) {
            for (int k = 0; k < ndim; ++k) {
                const int32_t v = coords[e * ndim + k];
                if (v < 0 || v >= dims[k]) return fail(nullptr, GCP_ERR_ARG, "coordinate out of range");
            }
            const float x = vals[e];
            if (!std::isfinite(x)) return fail(nullptr, GCP_ERR_ARG, "non-finite value");
            if ((loss == GCP_POISSON && x < 0.0f) || (loss == GCP_GAMMA && x <= 0.0f) ||
                (loss == GCP_BERNOULLI_LOGIT && x != 1.0f && x != 0.0f))
                return fail(nullptr, GCP_ERR_DOMAIN, "value outside the loss's domain");
        }
    }
    gcp_ctx *c = new (std::nothrow) gcp_ctx();
    if (!c) return fail(nullptr, GCP_ERR_OOM, "host allocation");
    gcp_status s = init_common(c, ndim, dims, rank, loss, opt);
    if (s) {
        destroy_buffers(c);
        delete c;
        return s;
    }
    if ((double)nnz > c->M) {
        destroy_buffers(c);
        delete c;
        return fail(nullptr, GCP_ERR_ARG, "more nonzeros than cells");
    }
    c->nnz = nnz;
    {
        std::vector<int64_t> counts((size_t)c->total_rows, 0);
        for (int64_t e = 0; e < nnz; ++e)
            for (int k = 0; k < ndim; ++k) ++counts[(size_t)(c->rowoff[k] + coords[e * ndim + k])];
        s = setup_hot_rows(c, counts);
        if (s) {
            destroy_buffers(c);
            delete c;
            return s;
        }
    }
    c->rec_words = gcpk::rec_words_for(ndim);
    const uint64_t cap = next_pow2((uint64_t)std::ceil((double)nnz / c->opt.hash_max_load)) < 4
                             ? 4
                             : next_pow2((uint64_t)std::ceil((double)nnz / c->opt.hash_max_load));
    c->hbmask = cap / 4 - 1;
    int32_t *dcoords = nullptr;
    float *dvals = nullptr;
    cudaError_t e;
    if ((e = cudaMalloc(&c->rec, (size_t)nnz * c->rec_words * 4)) || (e = cudaMalloc(&c->hkeys, cap * 8)) ||
        (e = cudaMalloc(&dcoords, (size_t)nnz * ndim * 4)) || (e = cudaMalloc(&dvals, (size_t)nnz * 4))) {
        cudaFree(dcoords);
        cudaFree(dvals);
        destroy_buffers(c);
        delete c;
        return cuda_fail(nullptr, e, "allocating nonzero storage");
    }
    if ((e = cudaMemsetAsync(c->hkeys, 0xFF, cap * 8, c->st)) ||
        (e = cudaMemcpyAsync(dcoords, coords, (size_t)nnz * ndim * 4, cudaMemcpyHostToDevice, c->st)) ||
        (e = cudaMemcpyAsync(dvals, vals, (size_t)nnz * 4, cudaMemcpyHostToDevice, c->st)) ||
        (e = gcpk::launch_build_records(dcoords, dvals, nnz, ndim, c->stride, c->rowoff, c->hot_slot,
                                        c->rec_words, c->rec, c->hkeys, c->hbmask, c->status, c->st)) ||
        (e = cudaStreamSynchronize(c->st))) {
        cudaFree(dcoords);
        cudaFree(dvals);
        destroy_buffers(c);
        delete c;
        return cuda_fail(nullptr, e, "building nonzero records");
    }
    cudaFree(dcoords);
    cudaFree(dvals);
    s = collect(c);
    if (s) {
        g_create_err = c->err;
        destroy_buffers(c);
        delete c;
        return s;
    }
    *out = c;
    return GCP_OK;
}

gcp_status gcp_create_dense(int32_t ndim, const int64_t *dims, const float *X, int32_t rank, int32_t loss,
                            const gcp_options *opt, gcp_ctx **out) {
    if (!out) return fail(nullptr, GCP_ERR_ARG, "out is NULL");
    *out = nullptr;
    if (!X) return fail(nullptr, GCP_ERR_ARG, "X is NULL");
    gcp_ctx *c = new (std::nothrow) gcp_ctx();
    if (!c) return fail(nullptr, GCP_ERR_OOM, "host allocation");
    gcp_options o;
    gcp_options_default(&o);
    if (opt) o = *opt;
    o.sampling = GCP_SAMPLING_UNIFORM;
    gcp_status s = init_common(c, ndim, dims, rank, loss, &o);
    if (s) {
        destroy_buffers(c);
        delete c;
        return s;
    }
    c->dense = true;
    c->nnz = (int64_t)c->M;
    s = setup_hot_rows(c, std::vector<int64_t>());
    if (s) {
        destroy_buffers(c);
        delete c;
        return s;
    }
    const size_t bytes = (size_t)c->M * 4;
    cudaError_t e;
    if ((e = cudaMalloc(&c->X, bytes)) ||
        (e = cudaMemcpyAsync(c->X, X, bytes, cudaMemcpyDefault, c->st))) {
        destroy_buffers(c);
        delete c;
        return cuda_fail(nullptr, e, "copying the dense tensor");
    }
    k_check_dense<<<4096, 256, 0, c->st>>>(c->X, (int64_t)c->M, c->loss, c->status);
    if ((e = cudaGetLastError()) != cudaSuccess) {
        destroy_buffers(c);
        delete c;
        return cuda_fail(nullptr, e, "checking the dense tensor");
    }
    s = collect(c);  // synchronises
    if (s) {
        g_create_err = c->err;
        destroy_buffers(c);
        delete c;
        return s;
    }
    *out = c;
    return GCP_OK;
}

void gcp_destroy(gcp_ctx *c) {
    if (!c) return;
    DeviceGuard g(c->device);
    cudaStreamSynchronize(c->st);
    destroy_buffers(c);
    delete c;
}

const char *gcp_last_error(const gcp_ctx *c) { return c ? c->err.c_str() : g_create_err.c_str(); }

int32_t gcp_ndim(const gcp_ctx *c) { return c ? c->d : 0; }
int32_t gcp_rank(const gcp_ctx *c) { return c ? c->R : 0; }
int64_t gcp_nnz(const gcp_ctx *c) { return c ? c->nnz : 0; }
int64_t gcp_num_params(const gcp_ctx *c) { return c ? c->total_rows * c->R : 0; }

gcp_status gcp_set_factors(gcp_ctx *c, const float *A) {
    if (!c || !A) return fail(c, GCP_ERR_ARG, "NULL argument");
    DeviceGuard g(c->device);
    return rows_in(c, 0, c->total_rows, A);
}

gcp_status gcp_set_factor(gcp_ctx *c, int32_t mode, const float *A_mode) {
    if (!c || !A_mode) return fail(c, GCP_ERR_ARG, "NULL argument");
    if (mode < 0 || mode >= c->d) return fail(c, GCP_ERR_ARG, "mode out of range");
    DeviceGuard g(c->device);
    return rows_in(c, c->rowoff[mode], c->dims[mode], A_mode);
}

gcp_status gcp_set_factor_list(gcp_ctx *c, const float *const *A_modes) {
    if (!c || !A_modes) return fail(c, GCP_ERR_ARG, "NULL argument");
    for (int k = 0; k < c->d; ++k)
        if (!A_modes[k]) return fail(c, GCP_ERR_ARG, "NULL factor pointer");
    DeviceGuard g(c->device);
    FactorSrc src{};
    bool device = true;
    for (int k = 0; k < c->d; ++k) {
        device = device && kernel_writable(c, A_modes[k], sizeof(float));
        src.A[k] = A_modes[k];
        src.rowoff[k] = c->rowoff[k];
    }
    src.rowoff[c->d] = c->total_rows;
    if (device) return stage_factors(c, src, 0, c->total_rows);
    for (int k = 0; k < c->d; ++k) {
        gcp_status s = rows_in(c, c->rowoff[k], c->dims[k], A_modes[k]);
        if (s) return s;
    }
    return GCP_OK;
}

gcp_status gcp_get_factors(gcp_ctx *c, float *A_out) {
    if (!c || !A_out) return fail(c, GCP_ERR_ARG, "NULL argument");
    DeviceGuard g(c->device);
    gcp_status s = rows_out(c, c->A, 0, c->total_rows, A_out);
    if (s) return s;
    return collect(c);
}

gcp_status gcp_reset_adam(gcp_ctx *c) {
    if (!c) return fail(c, GCP_ERR_ARG, "NULL context");
    DeviceGuard g(c->device);
    const size_t bytes = (size_t)c->total_rows * c->Rp * 4;
    GCP_CUDA(c, cudaMemsetAsync(c->B, 0, bytes, c->st));
    GCP_CUDA(c, cudaMemsetAsync(c->C, 0, bytes, c->st));
    return GCP_OK;
}

gcp_status gcp_sample(gcp_ctx *c, uint64_t iter, int64_t p, int64_t q, int32_t *idx_out, float *x_out,
                      float *w_out) {
    if (!c) return fail(c, GCP_ERR_ARG, "NULL context");
    DeviceGuard g(c->device);
    gcp_status s = check_counts(c, p, q);
    if (s) return s;
    double w_nz, w_z;
    weights(c, p, q, w_nz, w_z);
    GCP_CUDA(c, gcpk::launch_sample(sample_spec(c, iter, p, q), idx_out, x_out, w_out, (float)w_nz, (float)w_z,
                                    c->st));
    return GCP_OK;
}

gcp_status gcp_loss(gcp_ctx *c, uint64_t iter, int64_t p, int64_t q, double *loss_out) {
    if (!c || !loss_out) return fail(c, GCP_ERR_ARG, "NULL argument");
    DeviceGuard g(c->device);
    Outputs out;
    out.host = true;
    gcp_status s = run_fused(c, iter, p, q, false, nullptr, out);
    if (s) return s;
    s = host_result(c);
    *loss_out = c->h_loss[0];
    return s;
}

gcp_status gcp_loss_async(gcp_ctx *c, uint64_t iter, int64_t p, int64_t q, double *dloss_out) {
    if (!c || !dloss_out) return fail(c, GCP_ERR_ARG, "NULL argument");
    DeviceGuard g(c->device);
    Outputs out;
    out.dloss = dloss_out;
    return run_fused(c, iter, p, q, false, nullptr, out);
}

gcp_status gcp_grad(gcp_ctx *c, uint64_t iter, int64_t p, int64_t q, float *G_out, double *loss_out) {
    if (!c) return fail(c, GCP_ERR_ARG, "NULL context");
    DeviceGuard g(c->device);
    Outputs out;
    out.G = G_out;
    out.host = loss_out != nullptr;
    gcp_status s = run_fused(c, iter, p, q, true, nullptr, out);
    if (s || !loss_out) return s;
    s = host_result(c);
    *loss_out = c->h_loss[0];
    return s;
}

gcp_status gcp_grad_async(gcp_ctx *c, uint64_t iter, int64_t p, int64_t q, const float *dscale, float *G_out,
                          double *dloss_out) {
    if (!c) return fail(c, GCP_ERR_ARG, "NULL context");
    DeviceGuard g(c->device);
    Outputs out;
    out.G = G_out;
    out.dloss = dloss_out;
    return run_fused(c, iter, p, q, true, dscale, out);
}

gcp_status gcp_grad_factors_async(gcp_ctx *c, const float *const *A_modes, uint64_t iter, int64_t p, int64_t q,
                                  float *G_out, double *dloss_out) {
    if (!c || !A_modes) return fail(c, GCP_ERR_ARG, "NULL argument");
    FactorSrc src{};
    for (int k = 0; k < c->d; ++k) {
        if (!A_modes[k]) return fail(c, GCP_ERR_ARG, "NULL factor pointer");
        cudaPointerAttributes at{};
        if (cudaPointerGetAttributes(&at, A_modes[k]) != cudaSuccess ||
            (at.type != cudaMemoryTypeDevice && at.type != cudaMemoryTypeManaged) ||
            (at.type == cudaMemoryTypeDevice && at.device != c->device)) {
            cudaGetLastError();  // a host pointer is an argument error, not a sticky CUDA error
            return fail(c, GCP_ERR_ARG, "factor matrices must be device or managed memory of the context's device");
        }
        src.A[k] = A_modes[k];
        src.rowoff[k] = c->rowoff[k];
    }
    src.rowoff[c->d] = c->total_rows;
    DeviceGuard g(c->device);
    gcp_status s = check_counts(c, p, q);
    if (s) return s;
    if ((s = stage_factors(c, src, 0, c->total_rows))) return s;
    Outputs out;
    out.G = G_out;
    out.dloss = dloss_out;
    return run_fused(c, iter, p, q, G_out != nullptr, nullptr, out);
}

gcp_status gcp_scale_async(gcp_ctx *c, const double *dscale, const float *x, float *y, int64_t n) {
    if (!c) return fail(c, GCP_ERR_ARG, "NULL context");
    if (!dscale || !x || !y || n < 0) return fail(c, GCP_ERR_ARG, "NULL array or negative length");
    if (n == 0) return GCP_OK;
    DeviceGuard g(c->device);
    const int64_t want = (n + 255) / 256;
    k_scale<<<(unsigned)(want < 8192 ? want : 8192), 256, 0, c->st>>>(dscale, x, y, n);
    GCP_CUDA(c, cudaGetLastError());
    return GCP_OK;
}

gcp_status gcp_adam_step(gcp_ctx *c, const gcp_adam_params *prm, int64_t t) {
    if (!c || !prm) return fail(c, GCP_ERR_ARG, "NULL argument");
    DeviceGuard g(c->device);
    return adam_step_impl(c, prm, t);
}

gcp_status gcp_step(gcp_ctx *c, uint64_t iter, int64_t p, int64_t q, const gcp_adam_params *prm, int64_t t,
                    double *dloss_out) {
    if (!c || !prm) return fail(c, GCP_ERR_ARG, "NULL argument");
    if (t < 1) return fail(c, GCP_ERR_ARG, "Adam step t must be >= 1");
    if (!(prm->beta1 >= 0.0 && prm->beta1 < 1.0 && prm->beta2 >= 0.0 && prm->beta2 < 1.0 && prm->eps >= 0.0))
        return fail(c, GCP_ERR_ARG, "Adam parameters out of range");
    DeviceGuard g(c->device);
    return do_step(c, iter, p, q, prm, t, dloss_out);
}

gcp_status gcp_grad_norm(gcp_ctx *c, double *norm_out) {
    if (!c || !norm_out) return fail(c, GCP_ERR_ARG, "NULL argument");
    DeviceGuard g(c->device);
    const int64_t n = (int64_t)c->total_rows * c->Rp;  // padding columns hold zeros
    const int64_t want = (n + 255) / 256;
    const int nb = (int)std::max<int64_t>(1, std::min<int64_t>(want, 4 * (int64_t)c->max_blocks));
    // the loss partials are free once the gradient's loss is finished (stream order)
    k_sumsq_blocks<<<nb, 256, 0, c->st>>>(c->G, n, c->partials);
    k_sumsq_finish<<<1, 256, 0, c->st>>>(c->partials, nb, c->dloss + 2, c->status);
    GCP_CUDA(c, cudaGetLastError());
    GCP_CUDA(c, cudaMemcpyAsync(c->h_loss + 2, c->dloss + 2, sizeof(double), cudaMemcpyDeviceToHost, c->st));
    const gcp_status s = collect(c);  // synchronises
    *norm_out = c->h_loss[2];
    return s;
}

gcp_status gcp_sync(gcp_ctx *c) {
    if (!c) return fail(c, GCP_ERR_ARG, "NULL context");
    DeviceGuard g(c->device);
    return collect(c);
}

gcp_status gcp_fit(gcp_ctx *c, const gcp_fit_params *prm, gcp_fit_report *rep) {
    if (!c || !prm) return fail(c, GCP_ERR_ARG, "NULL argument");
    if (prm->iters < 1 || prm->max_epochs < 0 || prm->max_fails < 1 || !(prm->decay > 0.0))
        return fail(c, GCP_ERR_ARG, "bad fit parameters");
    DeviceGuard g(c->device);
    const size_t bytes = (size_t)c->total_rows * c->Rp * 4;
    if (!c->bk_A) {
        cudaError_t e;
        if ((e = cudaMalloc(&c->bk_A, bytes)) || (e = cudaMalloc(&c->bk_B, bytes)) ||
            (e = cudaMalloc(&c->bk_C, bytes)))
            return cuda_fail(c, e, "allocating fit backups");
    }
    gcp_fit_report r;
    std::memset(&r, 0, sizeof(r));
    const auto t0 = std::chrono::steady_clock::now();
    auto objective = [&](double &F) -> gcp_status {
        Outputs out;
        out.host = true;
        gcp_status s = run_fused(c, GCP_ITER_OBJECTIVE, prm->p_obj, prm->q_obj, false, nullptr, out);
        if (s) return s;
        s = host_result(c);
        F = c->h_loss[0];
        r.attempts_per_zero = prm->q_obj > 0 ? c->h_loss[1] / (double)prm->q_obj : 0.0;
        return s;
    };
    auto backup = [&](bool save) -> gcp_status {
        float *src[3] = {c->A, c->B, c->C}, *dst[3] = {c->bk_A, c->bk_B, c->bk_C};
        for (int i = 0; i < 3; ++i)
            GCP_CUDA(c, cudaMemcpyAsync(save ? dst[i] : src[i], save ? src[i] : dst[i], bytes,
                                        cudaMemcpyDeviceToDevice, c->st));
        return save ? GCP_OK : refresh_bf16(c);
    };
    double F = 0.0;
    gcp_status s = objective(F);
    if (s) return s;
    r.objective0 = F;
    double Fbest = F;
    int64_t t = 0, t_saved = 0, steps_run = 0;
    gcp_adam_params adam = prm->adam;
    uint64_t iter = prm->iter0;
    if ((s = backup(true))) return s;
    for (int epoch = 0; epoch < prm->max_epochs; ++epoch) {
        for (int it = 0; it < prm->iters; ++it) {
            if ((s = do_step(c, iter++, prm->p, prm->q, &adam, t + 1, nullptr))) return s;
            ++t;
            ++steps_run;
        }
        if ((s = objective(F))) return s;
        if (epoch < GCP_FIT_TRACE) r.trace[epoch] = F;
        r.epochs = epoch + 1;
        if (!(F < Fbest)) {  // failed epoch: restore and decay the rate
            if ((s = backup(false))) return s;
            t = t_saved;
            adam.lr *= prm->decay;
            if (++r.fails >= prm->max_fails) break;
        } else {
            Fbest = F;
            t_saved = t;
            if ((s = backup(true))) return s;
        }
    }
    GCP_CUDA(c, cudaStreamSynchronize(c->st));
    r.seconds = std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count();
    r.iterations = t;
    r.objective = Fbest;
    r.lr = adam.lr;
    r.grad_samples_per_s = r.seconds > 0 ? (double)(prm->p + prm->q) * (double)steps_run / r.seconds : 0.0;
    if (rep) *rep = r;
    return GCP_OK;
}

gcp_status gcp_profile(gcp_ctx *c, int32_t enable) {
    if (!c) return fail(c, GCP_ERR_ARG, "NULL context");
    c->prof = enable != 0;
    return GCP_OK;
}

gcp_status gcp_profile_read(gcp_ctx *c, double *kernel_ms, int64_t *launches) {
    if (!c || !kernel_ms || !launches) return fail(c, GCP_ERR_ARG, "NULL argument");
    DeviceGuard g(c->device);
    GCP_CUDA(c, cudaStreamSynchronize(c->st));
    double total = 0.0;
    for (size_t i = 0; i < c->prof_used; ++i) {
        float ms = 0.0f;
        GCP_CUDA(c, cudaEventElapsedTime(&ms, c->prof_ev[i].first, c->prof_ev[i].second));
        total += ms;
    }
    *kernel_ms = total;
    *launches = (int64_t)c->prof_used;
    c->prof_used = 0;
    return GCP_OK;
}

}  // extern "C"
