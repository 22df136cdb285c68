// Entry points of the fills (fill.cuh holds the persistent kernels, which
// fill_dna.cu, fill_dna_half.cu, fill_general.cu and fill_general_half.cu
// instantiate; fill_static.cuh those of the allocation-free forward fill).
#include "fill_static.cuh"

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

static __device__ __align__(256) uint8_t g_static_scratch[kStaticBytes];

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
            if (static_setup_dna() != cudaSuccess || static_setup_general() != cudaSuccess)
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
    const StaticGeom g = sc.dna4 ? static_geom_dna(alphabet) : static_geom_general(alphabet);
    auto launch = [&](bool rest, int grid) {
        if (sc.dna4) static_launch_dna(rest, bv, sc, scratch, g, grid, st);
        else static_launch_general(rest, bv, sc, scratch, g, grid, st);
    };
    // as many blocks as can be resident, as the array has slots for and as
    // there are chunks
    const int most = (int)(kStaticErrOff / (kStaticShortBytes * 2 * (kBlock / 32)));
    int first_grid = std::min(sms * std::max(g.first_per_sm, 1), most);
    first_grid = std::min(first_grid, (npairs - 1) / kStaticChunk + 1);
    launch(false, first_grid);
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
        launch(true, std::min(kStaticSlots / g.rest_warps, (npairs - 1) / g.rest_warps + 1));
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
