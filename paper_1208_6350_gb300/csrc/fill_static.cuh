// Kernels of the allocation-free forward fill (gsw_fill_static; fill.cu holds the
// entry point and the scratch, fill_static_dna.cu and fill_static_general.cu
// instantiate the kernels for 4-letter and other alphabets).
#pragma once
#include "fill.cuh"

namespace gsw {
namespace {

constexpr int kStaticMaxTarget = GSW_STATIC_MAX_TARGET;
constexpr size_t kStaticSlotBytes = (size_t)kStaticMaxTarget * sizeof(int32_t) + 2 * (size_t)kStaticMaxTarget * sizeof(int2);
static_assert(kStaticMaxTarget % 4 == 0 && kStaticSlotBytes % 16 == 0,
              "slots start on 16-byte boundaries (the fill's 8-byte max-array stores)");
constexpr int kStaticSlots = 152 * 4 * 2;  // pairs in flight of the second kernel, a warp each
// slots of the first kernel: the column maxima of one strip in 16-bit lanes
constexpr size_t kStaticShortBytes = (size_t)kStaticMaxTarget * sizeof(uint16_t);
constexpr size_t kStaticErrOff = kStaticSlotBytes * kStaticSlots;
constexpr size_t kStaticBytes = kStaticErrOff + 256;  // + the per-call counters
static_assert(kStaticBytes == GSW_STATIC_SCRATCH_BYTES, "header states the scratch size");

// counters of a call, zeroed before its kernels
struct StaticCounters {
    int32_t bad;   // pairs rejected
    int32_t next;  // chunks handed out
    int32_t rest;  // pairs left to the second kernel
};

// One pair by the P lanes of a group; false when its score left the lanes.
template <int P, int R, class L, bool DNA, bool ONE>
__device__ bool static_fill_pair(const BatchView &b, const Scoring &sc, int pair, uint32_t *wsm, int lane, int k,
                                 unsigned gmask, int gbase, uint8_t *cms, uint8_t *bnd) {
    gsw_result *rp = b.res + pair;
    Job job;
    job.q = b.q + b.q_off[pair];
    job.qs = 1;
    job.mrows = b.q_len[pair];
    job.t = b.t + b.t_off[pair];
    job.ts = 1;
    job.ncols = b.t_len[pair];
    job.stop_u = 0;
    job.cms = cms;
    job.bnd = bnd;
    const RingResult rr = ring_fill<P, R, L, DNA, ONE>(job, sc, wsm, k, gmask, gbase, lane);
    if (L::FOLD && rr.score > 32767 - sc.wmax) return false;  // refill in 32-bit lanes
    int s2 = 0, e2 = -1;
    const int end_t = rr.col, end_q = rr.score > 0 ? rr.row - rr.pad_top : -1;
    __syncwarp(gmask);
    secondary<P, L>(b, pair, job, end_t, job.mrows, k, gmask, &s2, &e2);
    if (k == 0) {
        rp->score1 = rr.score;
        rp->score2 = s2;
        rp->ref_end1 = end_t;
        rp->read_end1 = end_q;
        rp->ref_begin1 = -1;
        rp->read_begin1 = -1;
        rp->ref_end2 = e2;
        rp->cigar_len = 0;
        rp->cigar_off = -1;
        rp->flags = L::FOLD ? 0 : GSW_RES_S32;
        rp->reserved = 0;
    }
    return true;
}

// The checks gsw_align_batch makes before any fill, made here by each group
// before its pair's first access: lengths in [0, 2^24), offsets >= 0 and
// targets within the slot; then the letter codes.  Writes the record of a
// rejected or empty pair; true when the pair is to be filled.
template <int P>
__device__ __forceinline__ bool static_check(const BatchView &b, const Scoring &sc, int pair, int k, unsigned gmask,
                                             int32_t *bad_count) {
    const int m = b.q_len[pair], n = b.t_len[pair];
    bool bad = (uint32_t)m >= (1u << 24) || (uint32_t)n >= (1u << 24) || b.q_off[pair] < 0 || b.t_off[pair] < 0 ||
               ((b.flags & GSW_COLMAX) && b.colmax_off[pair] < 0) || n > kStaticMaxTarget;
    if (!bad) {
        const uint8_t *qp = b.q + b.q_off[pair], *tp = b.t + b.t_off[pair];
        int found = 0;
        for (int i = k; i < m; i += P) found |= qp[i] >= sc.A;
        for (int j = k; j < n; j += P) found |= tp[j] >= sc.A;
        bad = __any_sync(gmask, found) != 0;
    }
    const bool empty = !bad && (m == 0 || n == 0);
    if (k == 0 && (bad || empty)) {
        gsw_result *rp = b.res + pair;
        rp->score1 = 0; rp->score2 = 0; rp->ref_begin1 = -1; rp->ref_end1 = -1; rp->read_begin1 = -1;
        rp->read_end1 = -1; rp->ref_end2 = -1; rp->cigar_len = 0; rp->cigar_off = -1;
        rp->flags = bad ? kResInvalid : 0;
        rp->reserved = 0;
        if (bad) atomicOr(bad_count, 1);
    }
    if (empty && (b.flags & GSW_COLMAX))
        for (int j = k; j < n; j += P) b.colmax[b.colmax_off[pair] + j] = 0;
    return !bad && !empty;
}

// First kernel: the queries of one strip (at most kStaticRows) in 16-bit lanes.
// Their slots hold the column maxima alone, 2 KB, so the array has one for
// every group that can be resident, where slots that also fit 32-bit boundary
// rows (20 KB) allowed 4 warps per SM: 8,192 pairs of 100-250 x 300-1000 DNA
// letters 1.00 -> 0.56 ms, of 30-400 x 300-1000 2.88 -> 1.11 ms (strips of 320
// to 512 rows instead of two of 256), 100 of 30-400 x 100-900 0.50 -> 0.22 ms.
// A block takes kStaticChunk consecutive pairs (8: 0.55 ms, 16: 0.57, 24: 0.62),
// orders them by strip height and target length, and its warps take them two at
// a time (one per 16-lane group; both use the same row-word count R, because
// their profiles share the warp's interleaved shared-memory region).  Taller
// queries and scores beyond 16 bits are left to the second kernel, which runs
// only if some pair was.
constexpr int kStaticChunk = 8;
constexpr int kStaticRows = 512;
template <bool DNA>
__global__ void __launch_bounds__(kBlock, 3) k_fill_static(BatchView b, Scoring sc, uint8_t *scratch, int warp_words) {
    extern __shared__ __align__(16) uint32_t smem[];
    __shared__ int order[kStaticChunk], key[kStaticChunk], chunk, taken;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 4, k = lane & 15, gbase = g * 16;
    const unsigned gmask = 0xFFFFu << gbase;
    uint32_t *wsm = smem + (size_t)warp * warp_words;
    uint8_t *cms = scratch + (size_t)((blockIdx.x * (kBlock / 32) + warp) * 2 + g) * kStaticShortBytes;
    StaticCounters *cnt = reinterpret_cast<StaticCounters *>(scratch + kStaticErrOff);
    for (;;) {
        __syncthreads();
        if (threadIdx.x == 0) {
            chunk = atomicAdd(&cnt->next, 1);
            taken = 0;
        }
        __syncthreads();
        const long long base = (long long)chunk * kStaticChunk;
        if (base >= b.npairs) break;
        if (threadIdx.x < kStaticChunk) {
            const long long p = base + threadIdx.x;
            const int m = p < b.npairs ? b.q_len[p] : -1;
            // (lengths out of range sort anywhere: they are rejected below)
            key[threadIdx.x] = m < 0 ? -1 : (min(m, kStaticRows + 1) + 31) / 32 * 2048 + (b.t_len[p] & 2047);
        }
        __syncthreads();
        if (threadIdx.x < kStaticChunk) {
            int rank = 0;
            for (int x = 0; x < kStaticChunk; x++)
                rank += key[x] > key[threadIdx.x] || (key[x] == key[threadIdx.x] && x < (int)threadIdx.x);
            order[rank] = base + threadIdx.x < b.npairs ? (int)(base + threadIdx.x) : -1;
        }
        __syncthreads();
        for (;;) {
            int t = 0;
            if (lane == 0) t = atomicAdd(&taken, 2);
            t = __shfl_sync(0xFFFFFFFFu, t, 0);
            if (t >= kStaticChunk) break;
            const int pair = order[t + g];
            int m = 0, n = 0;
            bool run = false;
            if (pair >= 0) {
                if (b.q_len[pair] > kStaticRows) {
                    if (k == 0) cnt->rest = 1;  // (checked by the second kernel)
                } else {
                    run = static_check<16>(b, sc, pair, k, gmask, &cnt->bad);
                    m = b.q_len[pair];
                    n = b.t_len[pair];
                }
            }
            const int rows = __reduce_max_sync(0xFFFFFFFFu, run ? m : 0);
            const int most = __reduce_max_sync(0xFFFFFFFFu, run ? min(m, n) : 0);
            const bool half = half_fits(most, most, sc);
            bool ok = true;
            if (run) {
#define GSW_STATIC(R) \
    ok = half ? static_fill_pair<16, R, LH, DNA, true>(b, sc, pair, wsm, lane, k, gmask, gbase, cms, nullptr) \
              : static_fill_pair<16, R, L16, DNA, true>(b, sc, pair, wsm, lane, k, gmask, gbase, cms, nullptr)
                if (rows <= 64) GSW_STATIC(2);
                else if (rows <= 128) GSW_STATIC(4);
                else if (rows <= 192) GSW_STATIC(6);
                else if (rows <= 256) GSW_STATIC(8);
                else if (rows <= 320) GSW_STATIC(10);
                else if (rows <= 384) GSW_STATIC(12);
                else GSW_STATIC(16);
#undef GSW_STATIC
                if (!ok && k == 0) {
                    b.res[pair].flags = GSW_RES_S32 | kResPendingS32;
                    cnt->rest = 1;
                }
            }
            __syncwarp();
        }
    }
}

// Second kernel: queries of more than kStaticRows, a whole warp per pair, and
// pairs whose score left the 16-bit lanes.  Strips of 640 or 1,024 rows (256 in
// 32-bit lanes), in slots that hold the boundary rows of 32-bit lanes: two pairs a
// warp in strips of 256 rows took two to six times as many steps after the first
// kernel had ended (100 pairs of 500-1,000 x 1,000 DNA 1.12 -> 0.49 ms, 8,192 of
// 300-600 x 900 4.12 -> 1.69, 400 of 2,000-3,000 x 1,000 2.97 -> 0.98).
template <bool DNA>
__global__ void __launch_bounds__(kBlock) k_fill_static_rest(BatchView b, Scoring sc, uint8_t *scratch,
                                                             int warp_words) {
    extern __shared__ __align__(16) uint32_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int gwarp = blockIdx.x * (blockDim.x / 32) + warp;
    const int nwarps = gridDim.x * (blockDim.x / 32);
    constexpr unsigned ALL = 0xFFFFFFFFu;
    uint32_t *wsm = smem + (size_t)warp * warp_words;
    uint8_t *slot = scratch + (size_t)gwarp * kStaticSlotBytes;
    uint8_t *bnd = slot + (size_t)kStaticMaxTarget * sizeof(int32_t);
    StaticCounters *cnt = reinterpret_cast<StaticCounters *>(scratch + kStaticErrOff);
    for (long long at = gwarp; at < b.npairs; at += nwarps) {
        const int pair = (int)at;
        const int rows = b.q_len[pair];
        const bool tall = rows > kStaticRows;
        bool ok = tall || !(b.res[pair].flags & kResPendingS32) || (b.res[pair].flags & kResInvalid);
        if (tall && static_check<32>(b, sc, pair, lane, ALL, &cnt->bad)) {
            const int most = min(rows, b.t_len[pair]);
            const bool half = half_fits(most, most, sc);
#define GSW_STATIC(R, L, ONE) static_fill_pair<32, R, L, DNA, ONE>(b, sc, pair, wsm, lane, lane, ALL, 0, slot, bnd)
            if (rows > 1024) ok = GSW_STATIC(16, L16, false);
            else if (rows > 640) ok = half ? GSW_STATIC(16, LH, true) : GSW_STATIC(16, L16, true);
            else ok = half ? GSW_STATIC(10, LH, true) : GSW_STATIC(10, L16, true);
        }
        __syncwarp();
        if (!ok) GSW_STATIC(8, L32, false);
#undef GSW_STATIC
        __syncwarp();
    }
}

template <bool DNA>
StaticGeom static_geom(int alphabet) {
    StaticGeom g;
    g.first_warp = (size_t)prof_words(16, true, DNA, alphabet) * 32 * sizeof(uint32_t);
    g.first_smem = g.first_warp * (kBlock / 32);
    static OccupancyCache occ;
    g.first_per_sm = occ.get(k_fill_static<DNA>, kBlock, alphabet, g.first_smem, kStaticMaxSmem);
    // the second kernel's 16- or 32-bit profile, whichever is larger
    g.rest_warp = (size_t)std::max(prof_words(16, true, DNA, alphabet), prof_words(8, false, DNA, alphabet)) * 32 *
                  sizeof(uint32_t);
    g.rest_warps = std::max(1, std::min(4, (int)(kStaticMaxSmem / g.rest_warp)));
    return g;
}

template <bool DNA>
cudaError_t static_setup() {
    cudaError_t e = cudaFuncSetAttribute(k_fill_static<DNA>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStaticMaxSmem);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_fill_static_rest<DNA>, cudaFuncAttributeMaxDynamicSharedMemorySize, kStaticMaxSmem);
    return e;
}

template <bool DNA>
void static_launch(bool rest, const BatchView &b, const Scoring &sc, uint8_t *scratch, const StaticGeom &g, int grid,
                   cudaStream_t st) {
    if (rest)
        k_fill_static_rest<DNA><<<grid, g.rest_warps * 32, g.rest_warp * g.rest_warps, st>>>(b, sc, scratch,
                                                                                            (int)(g.rest_warp / 4));
    else
        k_fill_static<DNA><<<grid, kBlock, g.first_smem, st>>>(b, sc, scratch, (int)(g.first_warp / 4));
}

}  // namespace
}  // namespace gsw
