// gcp_mttkrp_det.cu -- deterministic all-mode sampled MTTKRP.
//
// The gradient of a sample set is G_n(i_n,:) = sum_s y_s prod_{k!=n}
// A_k(i_k,:) (Eq. gcp-gradient on the sampled gradient tensor).  The atomic
// variant adds these terms in whatever order the hardware applies the
// reductions.  This variant fixes the order, so G is bit-identical from run
// to run, in the spirit of the permutation-based MTTKRP of Sec. 3.1.2:
//   1. the fused kernel in materialize mode writes every sample's cell and
//      value y_s = w f'(x_s, m_s) (the non-fused gradient tensor) as one
//      record of RW words (i_0 .. i_{d-1}, y_s, zeros), so that a later
//      lookup of a sample reads one 16-byte vector (d <= 3);
//   2. per mode n, a stable LSD radix sort (7- or 8-bit digits, or one 10-bit
//      pass) orders (row, sample id) pairs by row i_n, ties in sample order.
//      The first pass of every mode is counted and scanned once for all
//      modes, and the modes are sorted side by side: pass p of every mode
//      that has one is a single launch per digit width over all their tiles,
//      so that it fills whole waves of resident blocks;
//   3. a chunked segmented reduction walks the sorted lists in chunks of
//      kChunk (64) positions, one chunk per group of lanes, recomputing the
//      Khatri-Rao row products, all modes of a sort group in one launch.  A
//      run of equal rows that lies inside one chunk is stored to
//      G directly; a run that crosses a chunk edge leaves one partial vector
//      per chunk it touches (in fixed slots: the right slot of its first
//      chunk, the left slots of the others);
//   4. a finishing pass sums each crossing run's partials in a fixed order
//      and stores the row.
// Every step has a fixed shape and order, so the result depends only on the
// inputs.
#include <cuda_bf16.h>

#include <utility>

#include "gcp_device.cuh"
#include "gcp_internal.h"

using namespace gcpdev;

namespace {

constexpr int kT = 256;            // threads per block
constexpr int kTile = 4096;        // keys per radix-sort block
constexpr int kChunk = 64;         // sorted positions per segmented-reduction chunk
constexpr int kScanBlock = 2048;   // elements per block of the multi-block scan
constexpr int kAhead = 4;          // partial vectors fetched ahead per lane group in the finishing pass

// --------------------------------------------------------------- radix sort
// One sort pass can sort several modes side by side (so that its blocks
// fill the GPU's waves): segment q sorts one mode's (key, sample id) pairs,
// read from `in`, or in a first pass from the records (keys at kin, kstride
// words apart, ids implied), into `out`.  Its digit counts start at obase in
// the count matrix, and `sub` is taken off its scanned offsets
// (k_radix_scatter).  Blocks [q * per, (q + 1) * per) of a launch work on
// segment q.
struct SortSeg {
    const int32_t *kin;
    const int2 *in;
    int2 *out;
    int64_t obase;
    uint32_t sub;
    int kstride;
};
struct SortSegs {
    int nseg;
    SortSeg s[GCP_MAX_NDIM];
};

// Segment q, read with constant indices only: a runtime index into a kernel
// parameter array would copy the whole array to local memory per thread.
__device__ __forceinline__ SortSeg pick_seg(const SortSegs &S, int q) {
    SortSeg r = S.s[0];
#pragma unroll
    for (int i = 1; i < GCP_MAX_NDIM; ++i)
        if (q == i) r = S.s[i];
    return r;
}

// Digits of NB = 128, 256 or 1024 values (7, 8 or 10 bits): the fewest passes
// and, among digits that need as many, the narrowest (digit_bits).  Segment
// q's count of digit d in tile t goes to hist[obase_q + d * ntiles + t].  A
// block counts kHistTiles consecutive tiles, so that it writes kHistTiles
// consecutive counts of each digit together.
constexpr int kHistTiles = 4;

// Digit width of a mode of `bits` key bits.
int digit_bits(int bits) {
    if (bits <= 7) return 7;
    if (bits <= 8) return 8;
    if (bits <= 10) return 10;  // one wide pass instead of two
    const int passes = (bits + 7) / 8;
    return 7 * passes >= bits ? 7 : 8;
}

template <int NB>
__global__ void k_radix_hist(const SortSegs SG, int64_t n, int shift, int32_t *__restrict__ hist, int ntiles) {
    __shared__ int h[kHistTiles][NB];
    for (int i = threadIdx.x; i < kHistTiles * NB; i += kT) (&h[0][0])[i] = 0;
    __syncthreads();
    const int per = (ntiles + kHistTiles - 1) / kHistTiles;
    const SortSeg sg = pick_seg(SG, blockIdx.x / per);
    const int2 *__restrict__ in = sg.in;
    const int t0 = (blockIdx.x % per) * kHistTiles;
    const int64_t first = (int64_t)t0 * kTile;
    constexpr int kB = 4;  // keys per tile loaded together, for every tile of the block
    for (int i0 = threadIdx.x; i0 < kTile; i0 += kB * kT) {
        int k[kHistTiles][kB];
#pragma unroll
        for (int g = 0; g < kHistTiles; ++g)
#pragma unroll
            for (int u = 0; u < kB; ++u) {
                const int64_t i = first + (int64_t)g * kTile + i0 + u * kT;
                k[g][u] = i < n ? in[i].x : -1;
            }
#pragma unroll
        for (int g = 0; g < kHistTiles; ++g)
#pragma unroll
            for (int u = 0; u < kB; ++u)
                if (k[g][u] >= 0) atomicAdd(&h[g][(k[g][u] >> shift) & (NB - 1)], 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kHistTiles * NB; i += kT) {
        const int d = i / kHistTiles, g = i % kHistTiles;
        if (t0 + g < ntiles) hist[sg.obase + (int64_t)d * ntiles + t0 + g] = h[g][d];
    }
}

// Words of a sample record: d coordinates and y, padded to 4, 8 or 16.
__host__ __device__ constexpr int rec_words(int d) { return d + 1 <= 4 ? 4 : (d + 1 <= 8 ? 8 : 16); }

// The first pass of every mode (shift 0) counted in one pass over the
// records: mode k's pass has nb[k] digits and its counts go to
// hist[base[k] + d * ntiles + t], the modes' count matrices side by side,
// so that one scan serves them all.  Shared counters of mode k start at
// soff[k].
struct FirstPlan {
    int d, rw;
    int nb[GCP_MAX_NDIM], soff[GCP_MAX_NDIM];
    int64_t base[GCP_MAX_NDIM];
};

__global__ void __launch_bounds__(kT) k_radix_hist_first(const int32_t *__restrict__ recs, int64_t n,
                                                          const FirstPlan F, int32_t *__restrict__ hist,
                                                          int ntiles, int G) {
    extern __shared__ int h[];  // [G][used]
    const int d = F.d;
    const int used = F.soff[d - 1] + F.nb[d - 1];
    for (int i = threadIdx.x; i < G * used; i += kT) h[i] = 0;
    __syncthreads();
    const int t0 = blockIdx.x * G;
    // kB records per thread at a time, their 16-byte vectors loaded together
    constexpr int kB = 4;
    const int nv = F.rw / 4;
    for (int g = 0; g < G; ++g) {
        const int64_t first = (int64_t)(t0 + g) * kTile;
        const int tile_n = first >= n ? 0 : (n - first < kTile ? (int)(n - first) : kTile);
        const int4 *__restrict__ r = reinterpret_cast<const int4 *>(recs + first * F.rw);
        int *hg = h + g * used;
        for (int i0 = threadIdx.x; i0 < tile_n; i0 += kB * kT)
            for (int v = 0; v < nv && 4 * v < d; ++v) {
                int4 q[kB];
#pragma unroll
                for (int u = 0; u < kB; ++u)
                    q[u] = i0 + u * kT < tile_n ? __ldg(r + (int64_t)(i0 + u * kT) * nv + v) : make_int4(0, 0, 0, 0);
#pragma unroll
                for (int u = 0; u < kB; ++u) {
                    if (i0 + u * kT >= tile_n) break;
                    const int c[4] = {q[u].x, q[u].y, q[u].z, q[u].w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int k = 4 * v + j;
                        if (k < d) atomicAdd(&hg[F.soff[k] + (c[j] & (F.nb[k] - 1))], 1);
                    }
                }
            }
    }
    __syncthreads();
    // G consecutive counts of a digit are written together
    for (int k = 0; k < d; ++k)
        for (int i = threadIdx.x; i < F.nb[k] * G; i += kT) {
            const int dg = i / G, g = i % G;
            if (t0 + g < ntiles) hist[F.base[k] + (int64_t)dg * ntiles + t0 + g] = h[g * used + F.soff[k] + dg];
        }
}

// Exclusive prefix sum of n ints of `in` (in = out scans in place), left in
// two parts: out[i] holds the scan within its block of kScanBlock elements
// and block_sums[i / kScanBlock] the scan of the block totals, so the full
// value is their sum (consumers add the two).  Each block scans its
// elements and records its total; the last block to finish (a ticket on
// `done`, which it clears again for the next scan) then scans the totals.
// Sums are taken modulo 2^32 (see k_radix_scatter).
__global__ void k_scan_blocks(const int32_t *in, int32_t *out, int64_t n, int32_t *block_sums, unsigned *done) {
    __shared__ int32_t warp_tot[kT / 32];
    __shared__ bool last;
    const int64_t base = (int64_t)blockIdx.x * kScanBlock + (int64_t)threadIdx.x * (kScanBlock / kT);
    int32_t v[kScanBlock / kT];
    int32_t sum = 0;
#pragma unroll
    for (int j = 0; j < kScanBlock / kT; ++j) {
        v[j] = base + j < n ? in[base + j] : 0;
        sum += v[j];
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    int32_t incl = sum;  // inclusive scan of the thread sums within the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int32_t t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[warp] = incl;
    __syncthreads();
    int32_t before = 0, block_total = 0;
    for (int w = 0; w < kT / 32; ++w) {
        if (w < warp) before += warp_tot[w];
        block_total += warp_tot[w];
    }
    int32_t run = before + incl - sum;
#pragma unroll
    for (int j = 0; j < kScanBlock / kT; ++j) {
        if (base + j < n) out[base + j] = run;
        run += v[j];
    }
    if (threadIdx.x == 0) {
        block_sums[blockIdx.x] = block_total;
        __threadfence();  // the total is visible before the ticket is taken
        last = atomicAdd(done, 1u) == gridDim.x - 1;
        if (last) __threadfence();  // and the other blocks' totals are seen after it
    }
    __syncthreads();
    if (!last) return;
    // the last block: exclusive scan of the gridDim.x totals, in place
    __shared__ int64_t part[kT];
    const int64_t nb = gridDim.x;
    const int64_t per = (nb + kT - 1) / kT;
    const int64_t lo = (int64_t)threadIdx.x * per, hi = lo + per < nb ? lo + per : nb;
    int64_t s = 0;
    for (int64_t i = lo; i < hi; ++i) s += __ldcg(block_sums + i);
    part[threadIdx.x] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        int64_t r = 0;
        for (int t = 0; t < kT; ++t) {
            const int64_t x = part[t];
            part[t] = r;
            r += x;
        }
        *done = 0u;
    }
    __syncthreads();
    int64_t r = part[threadIdx.x];
    for (int64_t i = lo; i < hi; ++i) {
        const int32_t x = __ldcg(block_sums + i);
        block_sums[i] = static_cast<int32_t>(static_cast<uint32_t>(r));
        r += x;
    }
}

void scan_two_part(const int32_t *in, int32_t *a, int64_t n, int32_t *block_sums, unsigned *done, cudaStream_t st) {
    const int64_t nb = (n + kScanBlock - 1) / kScanBlock;
    k_scan_blocks<<<(unsigned)nb, kT, 0, st>>>(in, a, n, block_sums, done);
}

// Stable scatter of one digit pass (NB digit values).  Each warp ranks its own
// kTile / 8 consecutive keys, 32 at a time in index order: lanes with equal
// digits find one another with ballots, take the digit's running count of
// the warp, and their first lane advances it.  One block-wide step then turns
// the warps' counts into local positions (warps in order, then digits), the
// pairs are placed in shared memory in that order, which leaves the tile
// sorted by digit, and are written out in order, so consecutive threads store
// consecutive pairs of a digit's run and the global writes are coalesced.
// Bound by that ranking, a chain of ballots and one shared counter per 32
// keys.  2^21 keys of two 14-bit modes, one 7-bit pass, 28 us; 41 us with
// match_any in place of the ballots (it takes a turn per distinct digit); 51
// us (8-bit) in a form that ranked 256 keys at a time over the whole block,
// with three barriers and a walk over all warps' counts of every digit per
// 256 keys.  The 10-bit pass of a 1000-row mode 30, 39 and 64 us.
// Block b sorts tile b % ntiles of segment b / ntiles.  The offset of digit
// d in this tile is offsets[obase + d * ntiles + tile] plus its block's
// sum, minus `sub`: the counts of the segments (modes) whose count matrices
// come first in a shared scan (each sums to n).  The sums are
// taken modulo 2^32, so the difference is exact even where the running
// total passes 2^31.
// Shared memory (dynamic): the tile's pairs, then per digit the global shift
// and one count per warp.
constexpr int kW = kT / 32;
constexpr int kRounds = kTile / kT;  // keys per lane

// Lanes of the warp whose digit (of NB values) equals the caller's: one
// ballot per bit.
template <int NB>
__device__ __forceinline__ unsigned same_digit(int digit) {
    unsigned peers = 0xFFFFFFFFu;
#pragma unroll
    for (int b = 1; b < NB; b <<= 1) {
        const unsigned set = __ballot_sync(0xFFFFFFFFu, digit & b);
        peers &= digit & b ? set : ~set;
    }
    return peers;
}

template <int NB>
constexpr size_t scatter_smem_bytes() {
    return (size_t)kTile * sizeof(int2) + (size_t)(NB + kW * NB + kW) * sizeof(int32_t);
}

template <int NB>
__global__ void __launch_bounds__(kT, NB <= 256 ? 4 : 3) k_radix_scatter(const SortSegs SG, int64_t n, int shift,
                                                      const int32_t *__restrict__ offsets,
                                                      const int32_t *__restrict__ offset_blocks, int ntiles) {
    const SortSeg sg = pick_seg(SG, blockIdx.x / ntiles);
    const int tile = blockIdx.x % ntiles;
    constexpr int DPT = NB >= kT ? NB / kT : 1;  // digits per thread (the first NB threads)
    extern __shared__ __align__(16) int2 s_kv[];
    int *gshift = reinterpret_cast<int *>(s_kv + kTile);  // [NB]
    int *wcount = gshift + NB;                            // [kW][NB]
    int *wsum = wcount + kW * NB;                         // [kW]
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t first = (int64_t)tile * kTile;
    const int tile_n = n - first < kTile ? (int)(n - first) : kTile;
    const int i0 = warp * (kTile / kW) + lane;  // this lane's first key in the tile
    const int32_t *__restrict__ kin = sg.kin;
    const int2 *__restrict__ in = sg.in;
    int *const mine = wcount + warp * NB;
    int key[kRounds];
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        const int i = i0 + 32 * r;
        key[r] = 0;
        if (i < tile_n) key[r] = in ? in[first + i].x : __ldg(kin + (first + i) * sg.kstride);
    }
    for (int d = lane; d < NB; d += 32) mine[d] = 0;
    __syncwarp();
    unsigned rank[kRounds / 2];  // among the warp's keys of the same digit (below 512), two to a word
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        const bool valid = i0 + 32 * r < tile_n;
        const int digit = (key[r] >> shift) & (NB - 1);
        const unsigned peers = same_digit<NB>(digit) & __ballot_sync(0xFFFFFFFFu, valid);
        const int below = __popc(peers & ((1u << lane) - 1u));
        int base = 0;
        if (valid) base = mine[digit];
        if (r & 1)
            rank[r / 2] |= (unsigned)(base + below) << 16;
        else
            rank[r / 2] = (unsigned)(base + below);
        __syncwarp();
        if (valid && below == 0) mine[digit] = base + __popc(peers);
        __syncwarp();
    }
    __syncthreads();
    // exclusive scan over the digits (thread t: digits DPT t .. DPT t + DPT -
    // 1) and, within a digit, over the warps
    int cnt[DPT][kW], tot[DPT], tsum = 0;
#pragma unroll
    for (int j = 0; j < DPT; ++j) {
        const int d = DPT * threadIdx.x + j;
        tot[j] = 0;
#pragma unroll
        for (int w = 0; w < kW; ++w) {
            cnt[j][w] = d < NB ? wcount[w * NB + d] : 0;
            tot[j] += cnt[j][w];
        }
        tsum += tot[j];
    }
    int incl = tsum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    int start = incl - tsum;
    for (int w = 0; w < warp; ++w) start += wsum[w];
#pragma unroll
    for (int j = 0; j < DPT; ++j) {
        const int d = DPT * threadIdx.x + j;
        if (d < NB) {
            const int64_t oi = sg.obase + (int64_t)d * ntiles + tile;
            const uint32_t off = (uint32_t)offsets[oi] + (uint32_t)offset_blocks[oi / kScanBlock] - sg.sub;
            gshift[d] = (int)off - start;
            int at = start;
#pragma unroll
            for (int w = 0; w < kW; ++w) {
                wcount[w * NB + d] = at;
                at += cnt[j][w];
            }
            start += tot[j];
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kRounds; ++r) {
        const int i = i0 + 32 * r;
        if (i < tile_n)
            s_kv[mine[(key[r] >> shift) & (NB - 1)] + (int)((rank[r / 2] >> (16 * (r & 1))) & 0xFFFFu)] =
                make_int2(key[r], in ? in[first + i].y : (int32_t)(first + i));
    }
    __syncthreads();
    int2 *__restrict__ out = sg.out;
    for (int i = threadIdx.x; i < tile_n; i += kT) {
        const int2 kv = s_kv[i];
        out[gshift[(kv.x >> shift) & (NB - 1)] + i] = kv;
    }
}

// ------------------------------------------------------ segmented reduction
// The modes m0, m0 + 1, ... of a sort group are reduced side by side: block
// row blockIdx.y works on mode m0 + blockIdx.y, so that one launch fills whole
// waves of resident blocks: 2^21 samples on 10^4 x 10^4 x 10^3 at rank 64 are
// 2.25 waves in each of three launches (234 us together), 6.7 in one (193 us).
struct SegSpec {
    int m0;
    int d, Rp, cols, log2L;
    int rowoff[GCP_MAX_NDIM];  // first rows of the modes in F and G
    const void *F;        // factors read by the kernels (FP32 or BF16)
    const int32_t *recs;  // sample records: d coordinates, y, padding (rec_words(d) words)
    float *G;
    const int2 *pairs;    // per mode of the group two arrays of n sorted (row, sample id) pairs
    unsigned parity;      // bit j: which of them holds mode m0 + j's order
    float *cvec;          // per mode of the group, partial vectors: two slots per chunk
    int64_t cstride;      // floats between the modes' partials
    int32_t *rowstart;    // per row of every mode, where its run starts
};

// What a block row of a reduction works on.
struct SegMode {
    int n_mode, rown;     // mode and its first row
    const int2 *kv;
    float *cvec;
    int32_t *rowstart;
};

__device__ __forceinline__ SegMode seg_mode(const SegSpec &P, int64_t n) {
    const int j = blockIdx.y;
    SegMode m;
    m.n_mode = P.m0 + j;
    m.rown = 0;
#pragma unroll
    for (int k = 0; k < GCP_MAX_NDIM; ++k)  // constant indices only
        if (k == m.n_mode) m.rown = P.rowoff[k];
    m.kv = P.pairs + (2 * j + ((P.parity >> j) & 1)) * n;
    m.cvec = P.cvec + j * P.cstride;
    m.rowstart = P.rowstart + m.rown;
    return m;
}

template <typename TF, int NQ>
__device__ __forceinline__ void load_cols(const TF *F, int off, const int (&col)[NQ], float (&o)[4 * NQ]) {
#pragma unroll
    for (int q = 0; q < NQ; ++q) Quad<TF>::load(F + off + col[q], o + 4 * q);
}

// Emit one run of equal keys: a run inside the chunk is final (stored to G),
// a run touching a chunk edge leaves the chunk's partial in its left slot
// (the run started earlier; also when it continues later) or its right slot
// (the run starts here and continues later).
template <int NQ>
__device__ __forceinline__ void emit_run(float *G, int Rp, int row_base, int key, const float (&acc)[4 * NQ],
                                         const int (&col)[NQ], bool before, bool after, int64_t chunk, float *cvec) {
    float *dst;
    if (!before && !after)
        dst = G + (int64_t)(row_base + key) * Rp;
    else
        dst = cvec + (2 * chunk + (before ? 0 : 1)) * Rp;
#pragma unroll
    for (int q = 0; q < NQ; ++q)
        *reinterpret_cast<float4 *>(dst + col[q]) = make_float4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
}

// Level 1: sorted sample ids of one mode -> G rows and edge carries.
// The group walks its chunk in batches of L positions.  Each lane first
// fetches one position's metadata (row key, then the sample's record: y_s
// and the coordinates that give the factor-row offsets), so the dependent
// id -> record lookups of a batch overlap; the positions are then taken in order, their metadata broadcast
// by shuffles and the factor rows of U positions gathered before any of
// them is accumulated.  Products and sums keep the sequential order.
template <typename TF, int COLS, int D>
__global__ void __launch_bounds__(kT, COLS == 8 && D >= 5 ? 2 : 3) k_seg_samples(const SegSpec P, int64_t n) {
    const SegMode M = seg_mode(P, n);
    const int2 *__restrict__ kv = M.kv;
    float *const cvec = M.cvec;
    int32_t *const rowstart = M.rowstart;
    constexpr int NQ = COLS / 4;
    constexpr int U0 = 32 / ((D - 1) * COLS);
    constexpr int U = U0 < 1 ? 1 : (U0 > 4 ? 4 : U0);  // positions gathered ahead
    const int lane = threadIdx.x & 31;
    const int L = 1 << P.log2L;
    const int glane = lane & (L - 1);
    const unsigned gmask = (L == 32) ? 0xFFFFFFFFu : (((1u << L) - 1u) << (lane & ~(L - 1)));
    const int64_t group = ((int64_t)blockIdx.x * kT + threadIdx.x) >> P.log2L;
    const int64_t ngroups = ((int64_t)gridDim.x * kT) >> P.log2L;
    const int64_t nchunks = (n + kChunk - 1) / kChunk;
    const int nm = M.n_mode;
    const TF *__restrict__ F = static_cast<const TF *>(P.F);
    constexpr int RW = rec_words(D);
    const int4 *__restrict__ recs = reinterpret_cast<const int4 *>(P.recs);
    int col[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) col[q] = q * (P.Rp >> 1) + 4 * glane;
    int roff[D - 1];  // first rows of the other modes (constant indices only)
#pragma unroll
    for (int j = 0; j < D - 1; ++j) roff[j] = j < nm ? P.rowoff[j] : P.rowoff[j + 1];
    const int rown = M.rown;
    for (int64_t c = group; c < nchunks; c += ngroups) {
        const int64_t lo = c * kChunk, hi = lo + kChunk < n ? lo + kChunk : n;
        const int len = (int)(hi - lo);
        float acc[COLS];
#pragma unroll
        for (int v = 0; v < COLS; ++v) acc[v] = 0.0f;
        int cur = kv[lo].x;
        bool before = lo > 0 && kv[lo - 1].x == cur;
        if (!before && glane == 0) rowstart[cur] = (int32_t)lo;  // a run starts at the chunk's start
        // the first batch's metadata: key and id, then the record
        int nkey = 0;
        int64_t nid = 0;
        int4 nrec[RW / 4];
        if (lo + glane < hi) {
            const int2 t = kv[lo + glane];
            nkey = t.x;
            nid = t.y;
        }
#pragma unroll
        for (int v = 0; v < RW / 4; ++v)
            nrec[v] = lo + glane < hi ? __ldg(recs + nid * (RW / 4) + v) : make_int4(0, 0, 0, 0);
        for (int b = 0; b < len; b += L) {
            // this lane's position of the batch (its metadata was fetched
            // during the previous batch): key, y and the D-1 row offsets of
            // the other modes (mode k < n at j = k, k > n at k-1)
            const int mkey = nkey;
            int w[RW];
#pragma unroll
            for (int v = 0; v < RW / 4; ++v) {
                w[4 * v] = nrec[v].x;
                w[4 * v + 1] = nrec[v].y;
                w[4 * v + 2] = nrec[v].z;
                w[4 * v + 3] = nrec[v].w;
            }
            const float my = __int_as_float(w[D]);
            int moff[D - 1];
#pragma unroll
            for (int j = 0; j < D - 1; ++j) moff[j] = (roff[j] + (j < nm ? w[j] : w[j + 1])) * P.Rp;
            // the next batch's key and id now; its record once the first
            // rows of this batch are on their way
            const int64_t pn = lo + b + L + glane;
            const bool has_next = pn < hi;
            if (has_next) {
                const int2 t = kv[pn];
                nkey = t.x;
                nid = t.y;
            }
            const int nb = len - b < L ? len - b : L;
            for (int t0 = 0; t0 < nb; t0 += U) {
                int key[U];
                float y[U], a[U][D - 1][COLS];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int t = t0 + u < nb ? t0 + u : nb - 1;  // group-uniform
                    key[u] = __shfl_sync(gmask, mkey, t, L);
                    y[u] = __shfl_sync(gmask, my, t, L);
#pragma unroll
                    for (int j = 0; j < D - 1; ++j)
                        load_cols<TF, NQ>(F, __shfl_sync(gmask, moff[j], t, L), col, a[u][j]);
                }
                if (t0 == 0)
#pragma unroll
                    for (int v = 0; v < RW / 4; ++v)
                        nrec[v] = has_next ? __ldg(recs + nid * (RW / 4) + v) : make_int4(0, 0, 0, 0);
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (t0 + u >= nb) break;
                    if (key[u] != cur) {
                        emit_run<NQ>(P.G, P.Rp, rown, cur, acc, col, before, false, c, cvec);
#pragma unroll
                        for (int v = 0; v < COLS; ++v) acc[v] = 0.0f;
                        cur = key[u];
                        before = false;
                        if (glane == 0) rowstart[cur] = (int32_t)(lo + b + t0 + u);  // a run starts here
                    }
                    float prod[COLS];
#pragma unroll
                    for (int v = 0; v < COLS; ++v) prod[v] = y[u];
#pragma unroll
                    for (int j = 0; j < D - 1; ++j)
#pragma unroll
                        for (int v = 0; v < COLS; ++v) prod[v] *= a[u][j][v];
#pragma unroll
                    for (int v = 0; v < COLS; ++v) acc[v] += prod[v];
                }
            }
        }
        const bool after = hi < n && kv[hi].x == cur;
        emit_run<NQ>(P.G, P.Rp, rown, cur, acc, col, before, after, c, cvec);
    }
}

// Finishing pass: the runs that cross chunk edges.  Lane l < kOwn of warp w
// checks chunk c = kOwn w + l: it owns a run if the chunk's first run began
// in an earlier chunk and ends in this one.  The run's first chunk c0 comes
// from the run's start position, which level 1 recorded per row (rowstart);
// its partials are the right slot of c0 and the left slots of c0 + 1 .. c (a
// chunk the run covers entirely uses its left slot), 1 + c - c0 vectors in
// all.  The warp takes its owned runs one by one: its 32 / L lane groups each
// add every (32 / L)-th partial in order, kAhead at a time, and the group
// sums are combined by a butterfly over the groups.  Runs of more than kLong
// partials (a hot row of skewed data has thousands) are left to the whole
// block, whose groups share them the same way before the warps' sums are
// added in order.  The order is fixed by (c0, c) alone, so the row is the
// same from run to run.
// Latency bound: each run is a chain of a few loads.  2^21 samples of the
// 4-way Zipf tensor at rank 32: 31 us a mode, against 167 us with a warp for
// every run, however long, and 32 chunks a warp.
constexpr int kOwn = 8;
constexpr int64_t kLong = 64;

// The sum of the partials gi, gi + ng, gi + 2 ng, ... of the run from chunk c0
// to c (lane group gi of ng).
template <int NQ>
__device__ __forceinline__ void sum_partials(const float *__restrict__ cvec, int Rp, int64_t c0, int64_t c, int gi,
                                             int ng, const int (&col)[NQ], float (&acc)[4 * NQ]) {
    const int64_t np = 1 + c - c0;
#pragma unroll
    for (int v = 0; v < 4 * NQ; ++v) acc[v] = 0.0f;
    for (int64_t k0 = gi; k0 < np; k0 += (int64_t)kAhead * ng) {
        float4 t[kAhead][NQ];
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            const int64_t k = k0 + (int64_t)u * ng;
            const int64_t slot = k < np ? (k == 0 ? 2 * c0 + 1 : 2 * (c0 + k)) : 2 * c;
#pragma unroll
            for (int q = 0; q < NQ; ++q) t[u][q] = *reinterpret_cast<const float4 *>(cvec + slot * Rp + col[q]);
        }
#pragma unroll
        for (int u = 0; u < kAhead; ++u) {
            if (k0 + (int64_t)u * ng >= np) break;
#pragma unroll
            for (int q = 0; q < NQ; ++q) {
                acc[4 * q] += t[u][q].x;
                acc[4 * q + 1] += t[u][q].y;
                acc[4 * q + 2] += t[u][q].z;
                acc[4 * q + 3] += t[u][q].w;
            }
        }
    }
}

template <int COLS>
__global__ void __launch_bounds__(kT) k_seg_finish(const SegSpec P, int64_t n) {
    const SegMode M = seg_mode(P, n);
    const int2 *__restrict__ kv = M.kv;
    const float *__restrict__ cvec = M.cvec;
    const int32_t *__restrict__ rowstart = M.rowstart;
    constexpr int NQ = COLS / 4;
    __shared__ int s_key[kW * kOwn];      // of a long run that ends in the block's chunk, else -1
    __shared__ int64_t s_c0[kW * kOwn];
    __shared__ float4 s_sum[kW][32];      // a warp's sum of a long run, one row (at most 128 floats)
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int L = 1 << P.log2L;
    const int glane = lane & (L - 1);
    const int grp = lane >> P.log2L, ngrp = 32 >> P.log2L;
    const int64_t nchunks = (n + kChunk - 1) / kChunk;
    const int64_t cw = ((int64_t)blockIdx.x * kW + warp) * kOwn;  // the warp's first chunk
    bool own = false;
    int mykey = -1;
    int64_t myc0 = 0;
    if (lane < kOwn && cw + lane < nchunks) {
        const int64_t cl = cw + lane;
        const int64_t lo = cl * kChunk, hi = lo + kChunk < n ? lo + kChunk : n;
        mykey = kv[lo].x;
        own = lo > 0 && kv[lo - 1].x == mykey &&            // the first run began earlier
              !(kv[hi - 1].x == mykey && hi < n && kv[hi].x == mykey);  // and ends in this chunk
        if (own) myc0 = __ldg(rowstart + mykey) / kChunk;
    }
    const bool big = own && cw + lane - myc0 >= kLong;
    if (lane < kOwn) {
        s_key[warp * kOwn + lane] = big ? mykey : -1;
        s_c0[warp * kOwn + lane] = myc0;
    }
    int col[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) col[q] = q * (P.Rp >> 1) + 4 * glane;
    float acc[COLS];
    auto over_groups = [&]() {  // butterfly over the warp's groups, fixed order
        for (int o = L; o < 32; o <<= 1)
#pragma unroll
            for (int v = 0; v < COLS; ++v) acc[v] += __shfl_xor_sync(0xFFFFFFFFu, acc[v], o);
    };
    for (unsigned owners = __ballot_sync(0xFFFFFFFFu, own && !big); owners; owners &= owners - 1) {
        const int j = __ffs(owners) - 1;
        const int key = __shfl_sync(0xFFFFFFFFu, mykey, j);
        const int64_t c0 = __shfl_sync(0xFFFFFFFFu, myc0, j);
        sum_partials<NQ>(cvec, P.Rp, c0, cw + j, grp, ngrp, col, acc);
        over_groups();
        if (grp == 0) {
            float *dst = P.G + (int64_t)(M.rown + key) * P.Rp;
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                *reinterpret_cast<float4 *>(dst + col[q]) =
                    make_float4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
        }
    }
    __syncthreads();
    for (int i = 0; i < kW * kOwn; ++i) {
        const int key = s_key[i];
        if (key < 0) continue;  // the same for the whole block
        sum_partials<NQ>(cvec, P.Rp, s_c0[i], (int64_t)blockIdx.x * kW * kOwn + i, warp * ngrp + grp, kW * ngrp, col,
                         acc);
        over_groups();
        if (grp == 0)
#pragma unroll
            for (int q = 0; q < NQ; ++q)
                s_sum[warp][col[q] >> 2] = make_float4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
        __syncthreads();
        if ((int)threadIdx.x < P.Rp >> 2) {
            float4 t = s_sum[0][threadIdx.x];
            for (int w = 1; w < kW; ++w) {
                const float4 v = s_sum[w][threadIdx.x];
                t.x += v.x;
                t.y += v.y;
                t.z += v.z;
                t.w += v.w;
            }
            reinterpret_cast<float4 *>(P.G + (int64_t)(M.rown + key) * P.Rp)[threadIdx.x] = t;
        }
        __syncthreads();
    }
}

int grid_for(int64_t items, int per_block) {
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > 65535) b = 65535;
    return (int)b;
}

}  // namespace

// Modes sorted side by side: as many as fit sort buffers of 1 GiB (each
// mode needs two key/id pairs of S ints), at least one.
static int det_group(const gcp_ctx *c, int64_t S) {
    const int64_t per_mode = 16 * (S > 0 ? S : 1);
    const int64_t g = ((int64_t)1 << 30) / per_mode;
    return (int)(g < 1 ? 1 : (g > c->d ? c->d : g));
}

// Scratch for the deterministic variant, grown on demand.  The scans'
// ticket comes first, so that it keeps its place (and its zero) whatever
// the sample count.
static gcp_status det_scratch(gcp_ctx *c, int64_t S, size_t *offs) {
    const int64_t ntiles = (S + kTile - 1) / kTile;
    const int64_t nchunk = (S + kChunk - 1) / kChunk + 1;
    const int64_t nfirst = (int64_t)1024 * c->d * ntiles;  // first-pass counts of all modes (at most)
    const int g = det_group(c, S);
    size_t o = 0;
    auto take = [&](size_t bytes) {
        const size_t at = o;
        o += (bytes + 255) & ~(size_t)255;
        return at;
    };
    offs[0] = take(4);                              // the scans' finishing ticket (zero between scans)
    offs[1] = take((size_t)S * rec_words(c->d) * 4);  // sample records
    offs[2] = take((size_t)g * 4 * S * 4);          // per mode of a group: two arrays of (key, id) pairs
    offs[3] = take((size_t)nfirst * 4);             // first-pass digit counts / offsets of every mode
    offs[4] = take((size_t)((nfirst + kScanBlock - 1) / kScanBlock + 1) * 4);  // their scan block sums
    offs[5] = take((size_t)g * 256 * ntiles * 4);   // later-pass digit counts / offsets of a group
    offs[6] = take((size_t)((g * 256 * ntiles + kScanBlock - 1) / kScanBlock + 1) * 4);  // their block sums
    offs[7] = take((size_t)g * 2 * nchunk * c->Rp * 4);  // per mode of a group, partial vectors: a left and a right slot per chunk
    offs[8] = take((size_t)c->total_rows * 4);      // start position of each row's run
    if (o > c->det_scratch_bytes) {
        cudaFree(c->det_scratch);
        c->det_scratch = nullptr;
        c->det_scratch_bytes = 0;
        cudaError_t e = cudaMalloc(&c->det_scratch, o);
        if (e != cudaSuccess) {
            c->err = std::string("allocating deterministic MTTKRP scratch: ") + cudaGetErrorString(e);
            return e == cudaErrorMemoryAllocation ? GCP_ERR_OOM : GCP_ERR_CUDA;
        }
        c->det_scratch_bytes = o;
        e = cudaMemsetAsync(c->det_scratch, 0, 4, c->st);
        if (e != cudaSuccess) {
            c->err = std::string("clearing deterministic MTTKRP scratch: ") + cudaGetErrorString(e);
            return GCP_ERR_CUDA;
        }
    }
    return GCP_OK;
}

#define DET_CUDA(call)                                                           \
    do {                                                                         \
        cudaError_t e_ = (call);                                                 \
        if (e_ != cudaSuccess) {                                                 \
            c->err = std::string(#call) + ": " + cudaGetErrorString(e_);         \
            return GCP_ERR_CUDA;                                                 \
        }                                                                        \
    } while (0)

template <typename TF, int D>
static void launch_seg_samples_d(const SegSpec &P, int cols, dim3 grid, int64_t n, cudaStream_t st) {
    if (cols == 8)
        k_seg_samples<TF, 8, D><<<grid, kT, 0, st>>>(P, n);
    else
        k_seg_samples<TF, 4, D><<<grid, kT, 0, st>>>(P, n);
}

template <typename TF>
static void launch_seg_samples(const SegSpec &P, int cols, dim3 grid, int64_t n, cudaStream_t st) {
    switch (P.d) {
        case 2: launch_seg_samples_d<TF, 2>(P, cols, grid, n, st); break;
        case 3: launch_seg_samples_d<TF, 3>(P, cols, grid, n, st); break;
        case 4: launch_seg_samples_d<TF, 4>(P, cols, grid, n, st); break;
        case 5: launch_seg_samples_d<TF, 5>(P, cols, grid, n, st); break;
        case 6: launch_seg_samples_d<TF, 6>(P, cols, grid, n, st); break;
        case 7: launch_seg_samples_d<TF, 7>(P, cols, grid, n, st); break;
        default: launch_seg_samples_d<TF, 8>(P, cols, grid, n, st); break;
    }
}

// The 1024-digit scatter needs more than the default 48 KB of dynamic
// shared memory; raised once per device.
static cudaError_t allow_wide_scatter() {
    static int done_dev = -1;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess || done_dev == dev) return e;
    e = cudaFuncSetAttribute(k_radix_scatter<1024>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)scatter_smem_bytes<1024>());
    if (e == cudaSuccess) done_dev = dev;
    return e;
}

gcp_status gcpk_det_grad(gcp_ctx *c, const gcpk::FusedSpec &f0, int *blocks) {
    const int64_t S = f0.s.p + f0.s.q;
    size_t offs[9];
    gcp_status s = det_scratch(c, S > 0 ? S : 1, offs);
    if (s) return s;
    char *base = static_cast<char *>(c->det_scratch);
    const int rw = rec_words(c->d);
    unsigned *ticket = reinterpret_cast<unsigned *>(base + offs[0]);
    int32_t *recs = reinterpret_cast<int32_t *>(base + offs[1]);
    int2 *sortbuf = reinterpret_cast<int2 *>(base + offs[2]);
    int32_t *histF = reinterpret_cast<int32_t *>(base + offs[3]);
    int32_t *bsumF = reinterpret_cast<int32_t *>(base + offs[4]);
    int32_t *histL = reinterpret_cast<int32_t *>(base + offs[5]);
    int32_t *bsumL = reinterpret_cast<int32_t *>(base + offs[6]);
    float *cvec = reinterpret_cast<float *>(base + offs[7]);
    int32_t *rowstart = reinterpret_cast<int32_t *>(base + offs[8]);
    cudaStream_t st = c->st;
    DET_CUDA(allow_wide_scatter());

    // 1. loss partials and the materialised gradient tensor, as records
    gcpk::FusedSpec f = f0;
    f.G = nullptr;
    f.Ycoord = recs;
    f.Yval = reinterpret_cast<float *>(recs + c->d);
    f.ystride = rw;
    f.vstride = rw;
    f.log2L = c->eval_log2L;
    DET_CUDA(gcpk::launch_fused_eval(f, c->Abf != nullptr, c->eval_cols, c->max_blocks, st, blocks));
    if (S == 0) return GCP_OK;

    // 2a. the first pass of every mode: counted and scanned once
    const int64_t ntiles = (S + kTile - 1) / kTile;
    int keybits[GCP_MAX_NDIM], dbits[GCP_MAX_NDIM], npass[GCP_MAX_NDIM], narrow = 7;
    FirstPlan FP{};
    FP.d = c->d;
    FP.rw = rw;
    int64_t nfirst = 0;
    for (int k = 0; k < c->d; ++k) {
        int bits = 1;
        while ((1ll << bits) < c->dims[k]) ++bits;
        keybits[k] = bits;
        dbits[k] = digit_bits(bits);
        if (dbits[k] == 8) narrow = 8;
    }
    for (int k = 0; k < c->d; ++k) {
        if (dbits[k] == 7) dbits[k] = narrow;  // one launch per pass for all modes but the wide ones
        FP.nb[k] = 1 << dbits[k];
        npass[k] = (keybits[k] + dbits[k] - 1) / dbits[k];
        FP.soff[k] = k ? FP.soff[k - 1] + FP.nb[k - 1] : 0;
        FP.base[k] = nfirst;
        nfirst += (int64_t)FP.nb[k] * ntiles;
    }
    const int used = FP.soff[c->d - 1] + FP.nb[c->d - 1];
    const int G = used <= 3072 ? kHistTiles : 1;  // at most 48 KB of counters
    k_radix_hist_first<<<(int)((ntiles + G - 1) / G), kT, (size_t)G * used * 4, st>>>(recs, S, FP, histF,
                                                                                     (int)ntiles, G);
    scan_two_part(histF, histF, nfirst, bsumF, ticket, st);
    DET_CUDA(cudaGetLastError());

    SegSpec P{};
    P.d = c->d;
    P.Rp = c->Rp;
    P.cols = c->cols;
    P.log2L = c->log2L;
    for (int k = 0; k < c->d; ++k) P.rowoff[k] = (int)c->rowoff[k];
    P.F = f0.F;
    P.recs = recs;
    P.G = c->G;
    P.pairs = sortbuf;
    P.cvec = cvec;
    P.cstride = 2 * ((S + kChunk - 1) / kChunk + 1) * (int64_t)c->Rp;
    P.rowstart = rowstart;
    const int lanes = 1 << c->log2L;
    const int group = det_group(c, S);
    // pair array of mode n (the j-th of its group) that pass p writes
    auto pairs_of = [&](int j, int p) { return sortbuf + ((int64_t)j * 2 + (p & 1)) * S; };
    bool joined = true;  // no side-stream work outstanding
    for (int m0 = 0; m0 < c->d; m0 += group) {
        const int m1 = m0 + group < c->d ? m0 + group : c->d;
        // 2b. stable LSD radix sort of sample ids by row, the modes of the
        // group side by side: pass p of every mode in one launch per digit
        // width
        for (int p = 0;; ++p) {
            SortSegs segs[3] = {};  // 128-, 256- and 1024-digit passes
            int nseg = 0;           // of this pass's own count (p > 0)
            int64_t ncount = 0;
            for (int n = m0; n < m1; ++n) {
                if (p >= npass[n]) continue;
                SortSegs &sg = segs[dbits[n] == 7 ? 0 : (dbits[n] == 8 ? 1 : 2)];
                SortSeg &q = sg.s[sg.nseg];
                q.kin = recs + n;
                q.kstride = rw;
                q.in = p == 0 ? nullptr : pairs_of(n - m0, p - 1);
                q.out = pairs_of(n - m0, p);
                if (p == 0) {  // offsets from the shared first-pass scan
                    q.obase = FP.base[n];
                    q.sub = (uint32_t)((uint64_t)n * (uint64_t)S);
                } else {       // offsets from this pass's own count
                    q.obase = ncount;
                    q.sub = (uint32_t)((uint64_t)nseg * (uint64_t)S);
                    ncount += (int64_t)FP.nb[n] * ntiles;
                    ++nseg;
                }
                ++sg.nseg;
            }
            if (segs[0].nseg + segs[1].nseg + segs[2].nseg == 0) break;
            if (p > 0) {  // later passes: counted over the previous pass's order
                const int per = (int)((ntiles + kHistTiles - 1) / kHistTiles);
                if (segs[0].nseg)
                    k_radix_hist<128><<<segs[0].nseg * per, kT, 0, st>>>(segs[0], S, 7 * p, histL, (int)ntiles);
                if (segs[1].nseg)
                    k_radix_hist<256><<<segs[1].nseg * per, kT, 0, st>>>(segs[1], S, 8 * p, histL, (int)ntiles);
                scan_two_part(histL, histL, ncount, bsumL, ticket, st);
            }
            const int32_t *offsets = p == 0 ? histF : histL, *blks = p == 0 ? bsumF : bsumL;
            // the 1024-digit launch (a first pass: there is no second) runs on
            // the side stream beside the narrower ones, so that each fills the
            // other's partial waves (both read only the records and the
            // first-pass offsets, and write their own modes' buffers)
            cudaStream_t wst = st;
            if (segs[2].nseg && segs[0].nseg + segs[1].nseg) {
                if (!c->det_side) {
                    DET_CUDA(cudaStreamCreateWithFlags(&c->det_side, cudaStreamNonBlocking));
                    DET_CUDA(cudaEventCreateWithFlags(&c->det_fork, cudaEventDisableTiming));
                    DET_CUDA(cudaEventCreateWithFlags(&c->det_join, cudaEventDisableTiming));
                }
                DET_CUDA(cudaEventRecord(c->det_fork, st));
                DET_CUDA(cudaStreamWaitEvent(c->det_side, c->det_fork, 0));
                wst = c->det_side;
            }
            if (segs[2].nseg)
                k_radix_scatter<1024><<<(int)(segs[2].nseg * ntiles), kT, scatter_smem_bytes<1024>(), wst>>>(
                    segs[2], S, 0, offsets, blks, (int)ntiles);
            if (segs[0].nseg)
                k_radix_scatter<128><<<(int)(segs[0].nseg * ntiles), kT, scatter_smem_bytes<128>(), st>>>(
                    segs[0], S, 7 * p, offsets, blks, (int)ntiles);
            if (segs[1].nseg)
                k_radix_scatter<256><<<(int)(segs[1].nseg * ntiles), kT, scatter_smem_bytes<256>(), st>>>(
                    segs[1], S, 8 * p, offsets, blks, (int)ntiles);
            DET_CUDA(cudaGetLastError());
            if (wst != st) {
                DET_CUDA(cudaEventRecord(c->det_join, wst));
                joined = false;
            }
        }
        if (!joined) {  // the wide modes' sort is done before their reduction
            DET_CUDA(cudaStreamWaitEvent(st, c->det_join, 0));
            joined = true;
        }
        P.m0 = m0;
        P.parity = 0;
        for (int n = m0; n < m1; ++n) P.parity |= (unsigned)((npass[n] - 1) & 1) << (n - m0);
        // 3. chunked segmented reduction over the sorted samples
        const int64_t nch = (S + kChunk - 1) / kChunk;
        const dim3 grid((unsigned)grid_for(nch * lanes, kT), (unsigned)(m1 - m0));
        if (c->Abf)
            launch_seg_samples<__nv_bfloat16>(P, c->cols, grid, S, st);
        else
            launch_seg_samples<float>(P, c->cols, grid, S, st);
        DET_CUDA(cudaGetLastError());
        // 4. the runs that cross chunk edges
        const dim3 fgrid((unsigned)((nch + kW * kOwn - 1) / (kW * kOwn)), (unsigned)(m1 - m0));
        if (c->cols == 8)
            k_seg_finish<8><<<fgrid, kT, 0, st>>>(P, S);
        else
            k_seg_finish<4><<<fgrid, kT, 0, st>>>(P, S);
        DET_CUDA(cudaGetLastError());
    }
    return GCP_OK;
}
