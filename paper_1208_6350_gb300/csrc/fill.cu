// Entry points of the fills (fill.cuh holds the kernels; fill_dna.cu and
// fill_general.cu instantiate the persistent ones for 4-letter and other
// alphabets) and the allocation-free forward fill.
#include "fill.cuh"

namespace gsw {

namespace {

// Calls f(class, geometry) for every class in fl.class_mask, heaviest first:
// the CTA kernel for queries of many strips, then the variants by rows per
// strip.  Stops when f returns false.
template <class F>
void each_class(const FillLaunch &fl, int sms, F f) {
    for (int c = kNumFillClasses - 1; c >= 0; c--) {
        if (!((fl.class_mask >> c) & 1u)) continue;  // no pair of the class
        const bool half = ((fl.half_mask >> c) & 1u) != 0;
        const ClassGeom g = fl.sc.dna4 ? (half ? fill_geom_dna_half(c, fl, sms) : fill_geom_dna(c, fl, sms))
                                       : (half ? fill_geom_general_half(c, fl, sms) : fill_geom_general(c, fl, sms));
        if (!f(c, g)) return;
    }
}

// No more blocks than the batch has pairs for (the CTA classes: a cluster per
// pair, whose warps share its strips).
void fit_pairs(const FillLaunch &fl, int c, ClassGeom &g) {
    const long long blocks = c >= kNumVariants ? (long long)fl.b.npairs * g.cluster
                                               : (fl.b.npairs + g.slots_per_block - 1) / std::max(1, g.slots_per_block);
    g.grid = (int)std::min<long long>(g.grid, std::max(1LL, blocks));
    if (g.grid < g.cluster) g.cluster = 1;
    g.grid -= g.grid % g.cluster;
}

// Every pair in flight has a slot: no more blocks than `bytes` hold.
bool fit_scratch(ClassGeom &g, size_t bytes) {
    const size_t per = (size_t)g.slots_per_block * (g.cm + g.bnd);
    if (g.grid > 0 && g.bytes(g.grid) > bytes)
        g.grid = (int)std::min<size_t>((size_t)g.grid, (bytes - std::min<size_t>(bytes, 256)) / per);
    if (g.grid < g.cluster) g.cluster = 1;
    g.grid -= g.grid % g.cluster;
    return g.grid > 0;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

}  // namespace

size_t fill_scratch_want(const FillLaunch &fl, int sms) {
    size_t sum = 0;
    each_class(fl, sms, [&](int c, ClassGeom g) {
        fit_pairs(fl, c, g);
        sum += align256(g.bytes(g.grid));
        return true;
    });
    return sum;
}

cudaError_t launch_fill(const FillLaunch &fl, int sms, cudaStream_t st, const SideStreams &aux) {
    struct Todo {
        int c;
        ClassGeom g;
        size_t at;
    } todo[kNumFillClasses];
    int n = 0;
    size_t sum = 0;
    each_class(fl, sms, [&](int c, ClassGeom g) {
        fit_pairs(fl, c, g);
        todo[n++] = Todo{c, g, sum};
        sum += align256(g.bytes(g.grid));
        return true;
    });
    // the classes whose pairs take longest first (strips x row words of a step)
    const ClassRows rows = fill_class_rows(fl.mode, fl.maxm, fl.sc, fl.class_mask);
    auto longest = [&](int c) {
        const int strips = (rows.most[c] + variant_rows(c) - 1) / variant_rows(c);
        return c >= kNumVariants ? INT_MAX : strips * (4 + variant_at(c).R);
    };
    std::stable_sort(todo, todo + n, [&](const Todo &a, const Todo &b) { return longest(a.c) > longest(b.c); });
    // classes side by side: the next one's blocks move in as one drains (a
    // batch of 20,000 reads of 100 to 250 nt is five launches, none of which
    // fills the chip)
    const bool side = n > 1 && aux.fork && sum <= fl.scr.bytes;
    SideFork fork(aux, st);
    cudaError_t e = fork.fork(side ? std::min(kSideStreams, n - 1) : 0);
    for (int i = 0; i < n && e == cudaSuccess; i++) {
        FillLaunch x = fl;
        ClassGeom &g = todo[i].g;
        if (side) x.scr.base = static_cast<char *>(fl.scr.base) + todo[i].at;
        else if (!fit_scratch(g, fl.scr.bytes)) return cudaErrorInvalidConfiguration;
        if (g.grid < 1) return cudaErrorInvalidConfiguration;
        x.scr.bnd_off = align256((size_t)g.grid * g.slots_per_block * g.cm);
        const int turn = i % (kSideStreams + 1);
        const cudaStream_t on = side && turn ? aux.s[turn - 1] : st;
        const int c = todo[i].c;
        const bool half = ((fl.half_mask >> c) & 1u) != 0;
        e = fl.sc.dna4 ? (half ? fill_launch_dna_half(c, x, g, on) : fill_launch_dna(c, x, g, on))
                       : (half ? fill_launch_general_half(c, x, g, on) : fill_launch_general(c, x, g, on));
    }
    const cudaError_t joined = fork.join();
    return e == cudaSuccess ? joined : e;
}

// ---------------------------------------------------------------------------
// Allocation-free forward fill (gsw_fill_static).  Its per-slot scratch (the
// column maxima and strip boundaries of a pair in flight) lives in a
// file-scope device array instead of context memory.
namespace {

constexpr int kStaticMaxTarget = GSW_STATIC_MAX_TARGET;
constexpr size_t kStaticSlotBytes = (size_t)kStaticMaxTarget * sizeof(int32_t) + 2 * (size_t)kStaticMaxTarget * sizeof(int2);
static_assert(kStaticMaxTarget % 4 == 0 && kStaticSlotBytes % 16 == 0,
              "slots start on 16-byte boundaries (the fill's 8-byte max-array stores)");
constexpr int kStaticWarps = 152 * 4;                 // warps of one launch
constexpr int kStaticSlots = kStaticWarps * 2;        // two pairs in flight per warp
// slots of the first kernel: the column maxima of one strip in 16-bit lanes
constexpr size_t kStaticShortBytes = (size_t)kStaticMaxTarget * sizeof(uint16_t);
constexpr size_t kStaticErrOff = kStaticSlotBytes * kStaticSlots;
constexpr size_t kStaticBytes = kStaticErrOff + 256;  // + the per-call counters
static_assert(kStaticBytes == GSW_STATIC_SCRATCH_BYTES, "header states the scratch size");

static __device__ __align__(256) uint8_t g_static_scratch[kStaticBytes];

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
__device__ __forceinline__ bool static_check(const BatchView &b, const Scoring &sc, int pair, int k, int P,
                                             unsigned gmask, int32_t *bad_count) {
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
                    run = static_check(b, sc, pair, k, 16, gmask, &cnt->bad);
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

// Second kernel: queries of several strips, and pairs whose score left the
// 16-bit lanes, in slots that hold the boundary rows of 32-bit lanes.  Warps
// take two pairs at a time (one per 16-lane group), grid-stride.
template <bool DNA>
__global__ void __launch_bounds__(kBlock) k_fill_static_rest(BatchView b, Scoring sc, uint8_t *scratch,
                                                             int warp_words) {
    extern __shared__ __align__(16) uint32_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 4, k = lane & 15, gbase = g * 16;
    const unsigned gmask = 0xFFFFu << gbase;
    const int gwarp = blockIdx.x * (blockDim.x / 32) + warp;
    const int nwarps = gridDim.x * (blockDim.x / 32);
    uint32_t *wsm = smem + (size_t)warp * warp_words;
    uint8_t *slot = scratch + (size_t)(gwarp * 2 + g) * kStaticSlotBytes;
    uint8_t *bnd = slot + (size_t)kStaticMaxTarget * sizeof(int32_t);
    StaticCounters *cnt = reinterpret_cast<StaticCounters *>(scratch + kStaticErrOff);
    for (long long base = gwarp * 2; base < b.npairs; base += nwarps * 2) {
        const int pair = (int)base + g;
        bool run = false, over = false;
        if (pair < b.npairs) {
            const bool tall = b.q_len[pair] > kStaticRows;
            over = !tall && (b.res[pair].flags & kResPendingS32) && !(b.res[pair].flags & kResInvalid);
            if (tall) run = static_check(b, sc, pair, k, 16, gmask, &cnt->bad);
        }
        bool ok = !over;
        if (run) ok = static_fill_pair<16, 8, L16, DNA, false>(b, sc, pair, wsm, lane, k, gmask, gbase, slot, bnd);
        __syncwarp();
        if (!ok) static_fill_pair<16, 8, L32, DNA, false>(b, sc, pair, wsm, lane, k, gmask, gbase, slot, bnd);
        __syncwarp();
    }
}

struct StaticSetup {
    bool done = false;
    uint8_t *ptr = nullptr;
    int sms = 0;
};
StaticSetup g_static_setup[64];
std::mutex g_static_mu;

}  // namespace

}  // namespace gsw

extern "C" int gsw_fill_static(int32_t npairs, const uint8_t *q, const int64_t *q_off, const int32_t *q_len,
                               const uint8_t *t, const int64_t *t_off, const int32_t *t_len,
                               int32_t max_target_len, const int8_t *matrix, int32_t alphabet, int32_t gap_open,
                               int32_t gap_extend, uint32_t flags, int32_t mask_len, gsw_result *results,
                               int32_t *colmax, const int64_t *colmax_off, void *stream) {
    using namespace gsw;
    if (npairs < 0) return set_err(GSW_EINVAL, "npairs < 0");
    if (flags & ~(uint32_t)GSW_COLMAX) return set_err(GSW_EINVAL, "flags other than GSW_COLMAX (0x%x)", flags);
    if (max_target_len < 0 || max_target_len > kStaticMaxTarget)
        return set_err(GSW_EINVAL, "max_target_len %d not in [0, %d]", max_target_len, kStaticMaxTarget);
    if (mask_len > (1 << 30)) return set_err(GSW_EINVAL, "mask_len too large");
    Scoring sc;
    {
        const int e = make_scoring(matrix, alphabet, gap_open, gap_extend, &sc);
        if (e != GSW_OK) return e;
    }
    if (npairs == 0) return GSW_OK;
    if (!q || !q_off || !q_len || !t || !t_off || !t_len || !results)
        return set_err(GSW_EINVAL, "NULL input or result pointer");
    if ((flags & GSW_COLMAX) && (!colmax || !colmax_off)) return set_err(GSW_EINVAL, "colmax output missing");
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return set_err(GSW_ECUDA, "no current device");
    // the second kernel's 16- or 32-bit profile, whichever is larger
    const size_t per_warp = (size_t)std::max(prof_words(8, true, sc.dna4 != 0, alphabet),
                                             prof_words(8, false, sc.dna4 != 0, alphabet)) * 32 * sizeof(uint32_t);
    int wpb = (int)((200u << 10) / per_warp);
    wpb = wpb > 4 ? 4 : (wpb < 1 ? 1 : wpb);
    const size_t smem = per_warp * wpb;
    const size_t short_warp = (size_t)prof_words(16, true, sc.dna4 != 0, alphabet) * 32 * sizeof(uint32_t);
    const size_t short_smem = short_warp * (kBlock / 32);
    uint8_t *scratch;
    int sms;
    {
        // once per device, with that device current: the device address of
        // the static scratch (the host-side symbol is only a stand-in)
        std::lock_guard<std::mutex> lk(g_static_mu);
        StaticSetup &su = g_static_setup[dev];
        if (!su.done) {
            void *ptr = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_scratch);
            if (e != cudaSuccess) return set_err(GSW_ECUDA, "scratch address: %s", cudaGetErrorString(e));
            for (const void *fn : {(const void *)k_fill_static<true>, (const void *)k_fill_static<false>,
                                   (const void *)k_fill_static_rest<true>, (const void *)k_fill_static_rest<false>})
                if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 << 10) != cudaSuccess)
                    return set_err(GSW_ECUDA, "kernel shared-memory limit");
            if (cudaDeviceGetAttribute(&su.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
                return set_err(GSW_ECUDA, "SM count");
            su.ptr = static_cast<uint8_t *>(ptr);
            su.done = true;
        }
        scratch = su.ptr;
        sms = su.sms;
    }
    BatchView bv;
    memset(&bv, 0, sizeof(bv));
    bv.q = q; bv.q_off = q_off; bv.q_len = q_len;
    bv.t = t; bv.t_off = t_off; bv.t_len = t_len;
    bv.res = results;
    bv.npairs = npairs;
    bv.flags = flags;
    bv.mask_len = mask_len;
    bv.colmax = colmax;
    bv.colmax_off = colmax_off;
    cudaStream_t st = (cudaStream_t)stream;
    // the counters must start at zero; the slots need no clearing
    if (cudaMemsetAsync(scratch + kStaticErrOff, 0, sizeof(StaticCounters), st) != cudaSuccess)
        return set_err(GSW_ECUDA, "clearing the counters");
    // as many blocks as can be resident, as the array has slots for and as
    // there are chunks
    static OccupancyCache occ[2];
    int per_sm = sc.dna4 ? occ[0].get(k_fill_static<true>, kBlock, alphabet, short_smem, 200 << 10)
                         : occ[1].get(k_fill_static<false>, kBlock, alphabet, short_smem, 200 << 10);
    const int most = (int)(kStaticErrOff / (kStaticShortBytes * 2 * (kBlock / 32)));
    int short_grid = std::min(sms * std::max(per_sm, 1), most);
    short_grid = std::min(short_grid, (npairs + kStaticChunk - 1) / kStaticChunk);
    const int grid = kStaticWarps / wpb;
    if (sc.dna4) k_fill_static<true><<<short_grid, kBlock, short_smem, st>>>(bv, sc, scratch, (int)(short_warp / 4));
    else k_fill_static<false><<<short_grid, kBlock, short_smem, st>>>(bv, sc, scratch, (int)(short_warp / 4));
    StaticCounters cnt = {};
    auto read_back = [&]() -> int {
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return set_err(GSW_ECUDA, "fill launch: %s", cudaGetErrorString(e));
        if (cudaMemcpyAsync(&cnt, scratch + kStaticErrOff, sizeof(cnt), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
            cudaStreamSynchronize(st) != cudaSuccess)
            return set_err(GSW_ECUDA, "counter readback");
        return GSW_OK;
    };
    {
        const int e = read_back();
        if (e != GSW_OK) return e;
    }
    if (cnt.rest) {  // the second kernel only where some pair was left to it
        if (sc.dna4) k_fill_static_rest<true><<<grid, wpb * 32, smem, st>>>(bv, sc, scratch, (int)(per_warp / 4));
        else k_fill_static_rest<false><<<grid, wpb * 32, smem, st>>>(bv, sc, scratch, (int)(per_warp / 4));
        const int e = read_back();
        if (e != GSW_OK) return e;
    }
    const int32_t err = cnt.bad;
    if (err)
        return set_err(GSW_EINVAL, "pairs with a length outside [0, 2^24), a target over %d letters, a negative "
                                   "offset or a letter code >= %d (records flagged GSW_RES_INVALID)",
                       kStaticMaxTarget, alphabet);
    return GSW_OK;
}
