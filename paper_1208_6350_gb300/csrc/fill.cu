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
    cudaError_t e = cudaSuccess;
    if (side) {
        if ((e = cudaEventRecord(aux.fork, st))) return e;
        for (int k = 0; k < 2 && k + 1 < n; k++)
            if ((e = cudaStreamWaitEvent(aux.s[k], aux.fork, 0))) return e;
    }
    for (int i = 0; i < n && e == cudaSuccess; i++) {
        FillLaunch x = fl;
        ClassGeom &g = todo[i].g;
        if (side) x.scr.base = static_cast<char *>(fl.scr.base) + todo[i].at;
        else if (!fit_scratch(g, fl.scr.bytes)) return cudaErrorInvalidConfiguration;
        if (g.grid < 1) return cudaErrorInvalidConfiguration;
        x.scr.bnd_off = align256((size_t)g.grid * g.slots_per_block * g.cm);
        const cudaStream_t on = side && i % 3 ? aux.s[i % 3 - 1] : st;
        const int c = todo[i].c;
        const bool half = ((fl.half_mask >> c) & 1u) != 0;
        e = fl.sc.dna4 ? (half ? fill_launch_dna_half(c, x, g, on) : fill_launch_dna(c, x, g, on))
                       : (half ? fill_launch_general_half(c, x, g, on) : fill_launch_general(c, x, g, on));
    }
    if (side)
        for (int k = 0; k < 2 && k + 1 < n; k++) {
            cudaError_t e2 = cudaEventRecord(aux.join[k], aux.s[k]);
            if (e2 == cudaSuccess) e2 = cudaStreamWaitEvent(st, aux.join[k], 0);
            if (e == cudaSuccess) e = e2;
        }
    return e;
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
constexpr size_t kStaticErrOff = kStaticSlotBytes * kStaticSlots;
constexpr size_t kStaticBytes = kStaticErrOff + 256;  // + the per-call error word
static_assert(kStaticBytes == GSW_STATIC_SCRATCH_BYTES, "header states the scratch size");

static __device__ __align__(256) uint8_t g_static_scratch[kStaticBytes];

template <int R, class L, bool DNA>
__device__ bool static_fill_pair(const BatchView &b, const Scoring &sc, int pair, uint32_t *wsm, int lane, int k,
                                 unsigned gmask, int gbase, uint8_t *slot) {
    gsw_result *rp = b.res + pair;
    Job job;
    job.q = b.q + b.q_off[pair];
    job.qs = 1;
    job.mrows = b.q_len[pair];
    job.t = b.t + b.t_off[pair];
    job.ts = 1;
    job.ncols = b.t_len[pair];
    job.stop_u = 0;
    job.cms = slot;
    job.bnd = slot + (size_t)kStaticMaxTarget * sizeof(int32_t);
    const RingResult rr = ring_fill<16, R, L, DNA>(job, sc, wsm, k, gmask, gbase, lane);
    if (L::FOLD && rr.score > 32767 - sc.wmax) return false;  // refill in 32-bit lanes
    int s2 = 0, e2 = -1;
    const int end_t = rr.col, end_q = rr.score > 0 ? rr.row - rr.pad_top : -1;
    __syncwarp(gmask);
    secondary<16, L>(b, pair, job, end_t, job.mrows, k, gmask, &s2, &e2);
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

// Warps take two pairs at a time (one per 16-lane group), grid-stride.  Both
// groups of a warp use the same row-word count R, because their profiles
// share the warp's interleaved shared-memory region; a group whose 16-bit
// fill overflowed refills afterwards in 32-bit lanes.
template <bool DNA>
__global__ void __launch_bounds__(kBlock) k_fill_static(BatchView b, Scoring sc, uint8_t *scratch, int warp_words) {
    extern __shared__ __align__(16) uint32_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = lane >> 4, k = lane & 15, gbase = g * 16;
    const unsigned gmask = 0xFFFFu << gbase;
    const int gwarp = blockIdx.x * (blockDim.x / 32) + warp;
    const int nwarps = gridDim.x * (blockDim.x / 32);
    uint32_t *wsm = smem + (size_t)warp * warp_words;
    uint8_t *slot = scratch + (size_t)(gwarp * 2 + g) * kStaticSlotBytes;
    int32_t *err = reinterpret_cast<int32_t *>(scratch + kStaticErrOff);
    for (int base = gwarp * 2; base < b.npairs; base += nwarps * 2) {
        const int pair = base + g;
        const bool has = pair < b.npairs;
        // the checks gsw_align_batch makes before any fill, made here by
        // each group before its pair's first access: lengths in [0, 2^24),
        // offsets >= 0 and targets within the slot; then the letter codes
        int m = 0, n = 0;
        bool bad = false;
        if (has) {
            m = b.q_len[pair];
            n = b.t_len[pair];
            bad = (uint32_t)m >= (1u << 24) || (uint32_t)n >= (1u << 24) || b.q_off[pair] < 0 || b.t_off[pair] < 0 ||
                  ((b.flags & GSW_COLMAX) && b.colmax_off[pair] < 0) || n > kStaticMaxTarget;
        }
        if (has && !bad) {
            const uint8_t *qp = b.q + b.q_off[pair], *tp = b.t + b.t_off[pair];
            int found = 0;
            for (int i = k; i < m; i += 16) found |= qp[i] >= sc.A;
            for (int j = k; j < n; j += 16) found |= tp[j] >= sc.A;
            bad = __any_sync(gmask, found) != 0;
        }
        const bool empty = has && !bad && (m == 0 || n == 0);
        const bool run = has && !bad && !empty;
        if (has && k == 0 && (bad || empty)) {
            gsw_result *rp = b.res + pair;
            rp->score1 = 0; rp->score2 = 0; rp->ref_begin1 = -1; rp->ref_end1 = -1; rp->read_begin1 = -1;
            rp->read_end1 = -1; rp->ref_end2 = -1; rp->cigar_len = 0; rp->cigar_off = -1;
            rp->flags = bad ? kResInvalid : 0;
            rp->reserved = 0;
            if (bad) atomicOr(err, 1);
        }
        if (empty && (b.flags & GSW_COLMAX))
            for (int j = k; j < n; j += 16) b.colmax[b.colmax_off[pair] + j] = 0;
        const int rows = __reduce_max_sync(0xFFFFFFFFu, run ? m : 0);
        bool ok = true;
        if (run) {
            if (rows <= 64) ok = static_fill_pair<2, L16, DNA>(b, sc, pair, wsm, lane, k, gmask, gbase, slot);
            else if (rows <= 128) ok = static_fill_pair<4, L16, DNA>(b, sc, pair, wsm, lane, k, gmask, gbase, slot);
            else if (rows <= 192) ok = static_fill_pair<6, L16, DNA>(b, sc, pair, wsm, lane, k, gmask, gbase, slot);
            else ok = static_fill_pair<8, L16, DNA>(b, sc, pair, wsm, lane, k, gmask, gbase, slot);
        }
        __syncwarp();
        if (!ok) static_fill_pair<8, L32, DNA>(b, sc, pair, wsm, lane, k, gmask, gbase, slot);
        __syncwarp();
    }
}

struct StaticSetup {
    bool done = false;
    uint8_t *ptr = nullptr;
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
    // (the 32-bit refill's profile may be the larger)
    const size_t per_warp = (size_t)std::max(prof_words(8, true, sc.dna4 != 0, alphabet),
                                             prof_words(8, false, sc.dna4 != 0, alphabet)) * 32 * sizeof(uint32_t);
    int wpb = (int)((200u << 10) / per_warp);
    wpb = wpb > 4 ? 4 : (wpb < 1 ? 1 : wpb);
    const size_t smem = per_warp * wpb;
    uint8_t *scratch;
    {
        // once per device, with that device current: the device address of
        // the static scratch (the host-side symbol is only a stand-in)
        std::lock_guard<std::mutex> lk(g_static_mu);
        StaticSetup &su = g_static_setup[dev];
        if (!su.done) {
            void *ptr = nullptr;
            const cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_scratch);
            if (e != cudaSuccess) return set_err(GSW_ECUDA, "scratch address: %s", cudaGetErrorString(e));
            if (cudaFuncSetAttribute(k_fill_static<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 << 10) !=
                    cudaSuccess ||
                cudaFuncSetAttribute(k_fill_static<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 << 10) !=
                    cudaSuccess)
                return set_err(GSW_ECUDA, "kernel shared-memory limit");
            su.ptr = static_cast<uint8_t *>(ptr);
            su.done = true;
        }
        scratch = su.ptr;
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
    // the error word must start at zero; the slots need no clearing
    if (cudaMemsetAsync(scratch + kStaticErrOff, 0, sizeof(int32_t), st) != cudaSuccess)
        return set_err(GSW_ECUDA, "clearing the error word");
    const int grid = kStaticWarps / wpb;
    if (sc.dna4) k_fill_static<true><<<grid, wpb * 32, smem, st>>>(bv, sc, scratch, (int)(per_warp / 4));
    else k_fill_static<false><<<grid, wpb * 32, smem, st>>>(bv, sc, scratch, (int)(per_warp / 4));
    {
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return set_err(GSW_ECUDA, "fill launch: %s", cudaGetErrorString(e));
    }
    int32_t err = 0;
    if (cudaMemcpyAsync(&err, scratch + kStaticErrOff, sizeof(int32_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return set_err(GSW_ECUDA, "error-word readback");
    if (err)
        return set_err(GSW_EINVAL, "pairs with a length outside [0, 2^24), a target over %d letters, a negative "
                                   "offset or a letter code >= %d (records flagged GSW_RES_INVALID)",
                       kStaticMaxTarget, alphabet);
    return GSW_OK;
}
