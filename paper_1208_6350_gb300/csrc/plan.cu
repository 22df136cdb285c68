// Work planning for the persistent fill launches, entirely on the device so
// that a batch needs no host round trip and the stage chain can be captured
// in a CUDA graph.  A counting sort groups pairs by fill class (how many
// query rows a strip covers; queries of many strips go to the CTA kernel)
// and, inside a class, by estimated cost (strips x steps) descending; the
// persistent kernels then hand out tasks heaviest class first, so long pairs
// start early and the tail is made of short ones.
#include "gsw_impl.cuh"

#include <atomic>
#include <climits>

namespace gsw {
namespace {

constexpr int kScanThreads = 1024;
// Batches of at most this many pairs are planned by one block.  Beyond, the
// block's turns over the pairs cost more than the two clears and three kernels of
// the chip-wide plan (whole calls of 30 x 60 DNA pairs with CIGARs, one block
// against the chip: 3,000 pairs 0.177 against 0.174 ms, 8,000 0.266 against
// 0.219, 16,000 0.411 against 0.304).
constexpr int kPlanSmall = 4096;
constexpr int kPlanFew = 2048;


__device__ __forceinline__ int cost_bin(long long cost) {
    // 32 bins per doubling of cost, descending order inside a variant
    float lg = log2f((float)(cost < 1 ? 1 : cost));
    int bin = (int)(lg * 32.0f);
    bin = bin < 0 ? 0 : (bin > kPlanBinsPerVariant - 1 ? kPlanBinsPerVariant - 1 : bin);
    return kPlanBinsPerVariant - 1 - bin;
}

// Sort key of pair p (class, then cost bin, descending), -1: not in the launch.
__device__ int plan_key(const BatchView &b, const Scoring &sc, int32_t mode, int p) {
    int rows, cols, v;
    if (mode == kFillForward) {
        rows = b.q_len[p];
        cols = b.t_len[p];
        if (b.flags & GSW_FORCE_S32) v = (cols > 0 && long_pair(rows, true, sc.dna4)) ? kClassLong32 : kVarS32;
        else v = (cols > 0 && rows > 0) ? pick_class16(rows, sc) : 0;  // (any class writes an empty pair's record)
        if (cta_pair(v, rows, cols, sc, false)) v = kClassLong16;
    } else if (mode == kFillRerun) {
        if (!(b.res[p].flags & kResPendingS32)) return -1;
        rows = b.q_len[p];
        cols = b.t_len[p];
        v = long_pair(rows, true, sc.dna4) ? kClassLong32 : kVarS32;
    } else if (mode == kFillReverse) {
        // the ring fill takes the reverse of pairs whose band is too wide or
        // too long for one thread
        const gsw_result r = b.res[p];
        if (r.score1 <= 0 || (r.flags & kResInternal)) return -1;
        rows = r.read_end1 + 1;
        const int wrev = reverse_band_width(r.read_end1, r.score1, sc);
        if (!small_batch(b) && wrev >= 0 && wrev <= kBandMaxRevWidth && rows <= kBandMaxRows) {
            return -1;
        }
        cols = reverse_window(r.read_end1, r.ref_end1, r.score1, sc);
        // a query of several strips reverses in the CTA kernel: its strips run
        // concurrently, so the stop at the first column reaching score1 (often
        // a few dozen columns into a window of thousands) ends every strip,
        // where a group would finish the upper strips over the whole window
        // before the last one starts (4-letter DNA: a general alphabet's CTA
        // holds 4 warps per SM)
        v = pick_class_reverse(rows, (r.flags & GSW_RES_S32) != 0, sc);
        if (cta_pair(v, rows, cols, sc, true)) v = kClassLong16;
    } else if (mode == kPlanTrace) {
        gsw_result r = b.res[p];
        if (small_batch(b) && r.score1 > 0 && !(r.flags & kResInternal)) {
            // a small batch has no band stage: all its pairs come here
            r.flags |= r.read_begin1 < 0 ? kResInternal : kResPendingTrace;  // (the ring reverse took every pair)
            b.res[p].flags = r.flags;
        }
        if (!wants_trace(r)) return -1;
        const int la = r.read_end1 - r.read_begin1 + 1, lb = r.ref_end1 - r.ref_begin1 + 1;
        int dlo, dhi;
        // 0-3: anti-diagonal warp kernel (<= 64/128/256/512 diagonals); 4:
        // wider bands, the CTA strip kernel; 5-8: the 16-bit rectangle
        const int cls = t16_launch_class(trace_class(la, lb, r.score1, sc, small_batch(b), &dlo, &dhi), la, sc.dna4 != 0);
        const int width = dhi - dlo + 1;
        long long cost = (long long)(la + lb + 1) * ((width + 31) / 32);
        if (cls >= kTraceT16First) {
            const T16Shape shape = t16_shape(cls - kTraceT16First, sc.dna4 != 0);
            cost = (long long)shape.strips(la) * shape.steps(lb);
        }
        return cls * kPlanBinsPerVariant + cost_bin(cost);
    } else {
        // kPlanBand: classes 0/1/2 = band width <= 8/16/32 diagonals
        const gsw_result r = b.res[p];
        if (r.score1 <= 0 || (r.flags & kResInternal)) return -1;
        int width;
        if (r.read_begin1 < 0) {
            const int wrev = reverse_band_width(r.read_end1, r.score1, sc);
            rows = r.read_end1 + 1;
            width = wrev < 0 ? INT_MAX : wrev;
            if (width > kBandMaxRevWidth || rows > kBandMaxRows) {
                b.res[p].flags |= kResInternal;  // the ring reverse should have taken it
                return -1;
            }
        } else {
            if (!(b.flags & GSW_CIGAR)) return -1;
            const int la = r.read_end1 - r.read_begin1 + 1, lb = r.ref_end1 - r.ref_begin1 + 1;
            int dlo, dhi;
            width = band_range(la, lb, r.score1, sc, &dlo, &dhi);
            rows = la;
            if (small_batch(b) || width > kBandMaxWidth || rows > kBandMaxRows) {
                b.res[p].flags |= kResPendingTrace;
                return -1;
            }
        }
        const int cls = width <= 8 ? 0 : (width <= 16 ? 1 : 2);
        return cls * kPlanBinsPerVariant + cost_bin(rows);
    }
    const Variant var = variant_at(v);
    const int sp = variant_rows(v);
    const long long strips = rows <= 0 ? 1 : (rows + sp - 1) / sp;
    const long long steps = (long long)cols + (var.s32 ? var.P : 2 * var.P);
    return v * kPlanBinsPerVariant + cost_bin(strips * steps);
}

// Counts and places of equal keys of a warp go to their bin in one atomic: a
// batch of equal shapes (all-vs-all overlaps) has one bin, whose atomics one by
// one took 2.8 ms for 4.2 M pairs, twice.
__global__ void k_plan_keys(BatchView b, Scoring sc, int32_t mode, int32_t *keys, int32_t *hist) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int key = p < b.npairs ? plan_key(b, sc, mode, p) : -1;
    if (p < b.npairs) keys[p] = key;
    const unsigned same = __match_any_sync(0xFFFFFFFFu, key);
    if (key >= 0 && (int)(threadIdx.x & 31) == __ffs(same) - 1) atomicAdd(&hist[key], __popc(same));
}

// Exclusive scan of `hist` (kPlanBins >> SHIFT counts) by a block of
// kScanThreads, in place or into binoff; then the class boundaries and task
// ranges.
template <int SHIFT>
__device__ void plan_scan(const int32_t *hist, int32_t *binoff, int32_t *var_start, int32_t *task_lo,
                          int32_t *task_hi, int32_t *ntasks, int32_t *head) {
    constexpr int BINS = kPlanBins >> SHIFT, PER = BINS / kScanThreads;
    static_assert(BINS % kScanThreads == 0 && (SHIFT > 0 || PER % 4 == 0), "bins");
    const int tid = threadIdx.x;
    int32_t loc[PER];
    int32_t sum = 0;
    if constexpr (SHIFT == 0) {
#pragma unroll
        for (int i = 0; i < PER; i += 4) {
            const int4 v = *reinterpret_cast<const int4 *>(hist + tid * PER + i);
            loc[i] = sum;
            loc[i + 1] = loc[i] + v.x;
            loc[i + 2] = loc[i + 1] + v.y;
            loc[i + 3] = loc[i + 2] + v.z;
            sum = loc[i + 3] + v.w;
        }
    } else {
#pragma unroll
        for (int i = 0; i < PER; i++) {
            loc[i] = sum;
            sum += hist[tid * PER + i];
        }
    }
    // inclusive scan of the threads' sums: within each warp by shuffles,
    // then over the warp totals by the first warp
    static_assert(kScanThreads == 32 * 32, "one warp scans the warp totals");
    __shared__ int32_t wsum[32];
    __shared__ int32_t starts[kNumFillClasses + 1];
    const int lane = tid & 31, warp = tid >> 5;
    int32_t incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const int32_t v = __shfl_up_sync(0xFFFFFFFFu, incl, d);
        if (lane >= d) incl += v;
    }
    if (lane == 31) wsum[warp] = incl;
    __syncthreads();
    if (warp == 0) {
        int32_t w = wsum[lane];
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t v = __shfl_up_sync(0xFFFFFFFFu, w, d);
            if (lane >= d) w += v;
        }
        wsum[lane] = w;
    }
    __syncthreads();
    const int32_t base = incl + (warp > 0 ? wsum[warp - 1] : 0) - sum;
    if constexpr (SHIFT == 0) {
#pragma unroll
        for (int i = 0; i < PER; i += 4)
            *reinterpret_cast<int4 *>(binoff + tid * PER + i) =
                make_int4(base + loc[i], base + loc[i + 1], base + loc[i + 2], base + loc[i + 3]);
    } else {
#pragma unroll
        for (int i = 0; i < PER; i++) binoff[tid * PER + i] = base + loc[i];
    }
    constexpr int OF_CLASS = kPlanBinsPerVariant >> SHIFT;
#pragma unroll
    for (int i = 0; i < PER; i++)
        if ((tid * PER + i) % OF_CLASS == 0) starts[(tid * PER + i) / OF_CLASS] = base + loc[i];
    if (tid == kScanThreads - 1) starts[kNumFillClasses] = base + sum;
    __syncthreads();
    // the classes' task ranges (heaviest class first), a lane per class
    static_assert(kNumFillClasses < 32, "a lane per class");
    if (warp == 0) {
        const int v = kNumFillClasses - 1 - lane;
        int32_t tasks = 0;
        if (v >= 0) {
            const int per = 32 / variant_at(v).P;
            tasks = (starts[v + 1] - starts[v] + per - 1) / per;
        }
        int32_t upto = tasks;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int32_t x = __shfl_up_sync(0xFFFFFFFFu, upto, d);
            if (lane >= d) upto += x;
        }
        if (v >= 0) {
            task_lo[v] = upto - tasks;
            task_hi[v] = upto;
            head[v] = 0;
        }
        if (v == 0) *ntasks = upto;
        if (lane <= kNumFillClasses) var_start[lane] = starts[lane];
    }
}

__global__ void __launch_bounds__(kScanThreads) k_plan_scan(const int32_t *hist, int32_t *binoff,
                                                             int32_t *var_start, int32_t *task_lo,
                                                             int32_t *task_hi, int32_t *ntasks, int32_t *head) {
    plan_scan<0>(hist, binoff, var_start, task_lo, task_hi, ntasks, head);
}

// The whole plan of a small batch by one block, its bins in shared memory: one
// launch instead of two clears and three kernels (about 25 us a plan, four or
// five plans a call).  SHIFT: 8 cost bins in one (4 per doubling) for batches
// that leave the chip part empty, where a finer order buys nothing (1,000 pairs:
// 8.0, 8.6 and 11.2 us a plan -> 6.1, 6.8 and 9.7).
template <int SHIFT>
__global__ void __launch_bounds__(kScanThreads) k_plan_small(BatchView b, Scoring sc, int32_t mode, PlanBuffers pb,
                                                              unsigned long long *need) {
    extern __shared__ __align__(16) int32_t bins[];
    __shared__ unsigned most[kNeedWords];
    if (threadIdx.x < kNeedWords) most[threadIdx.x] = 0;
    for (int i = threadIdx.x; i < (kPlanBins >> SHIFT) / 4; i += kScanThreads) reinterpret_cast<int4 *>(bins)[i] = make_int4(0, 0, 0, 0);
    __syncthreads();
    for (int p = threadIdx.x; p < b.npairs; p += kScanThreads) {
        const int key = plan_key(b, sc, mode, p);
        pb.keys[p] = key;
        if (key >= 0) atomicAdd(&bins[key >> SHIFT], 1);
        if (need && key >= 0) {
            unsigned v[kNeedWords] = {};
            trace_needs(b.res[p], sc, small_batch(b), v);
#pragma unroll
            for (int k = 0; k < kNeedWords; k++) {
                if (k == kNeedMask) atomicOr(&most[k], v[k]);
                else if (v[k]) atomicMax(&most[k], v[k]);
            }
        }
    }
    __syncthreads();
    if (need && threadIdx.x < kNeedWords) need[threadIdx.x] = most[threadIdx.x];
    plan_scan<SHIFT>(bins, bins, pb.var_start, pb.task_lo, pb.task_hi, pb.ntasks, pb.head);
    __syncthreads();
    for (int p = threadIdx.x; p < b.npairs; p += kScanThreads) {
        const int key = pb.keys[p];
        if (key >= 0) pb.order[atomicAdd(&bins[key >> SHIFT], 1)] = p;
    }
}

__global__ void k_plan_scatter(int32_t npairs, const int32_t *keys, const int32_t *binoff, int32_t *cursor,
                               int32_t *order) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
    const int key = p < npairs ? keys[p] : -1;
    const unsigned same = __match_any_sync(0xFFFFFFFFu, key);
    const int first = __ffs(same) - 1;
    int at = 0;
    if (key >= 0 && lane == first) at = binoff[key] + atomicAdd(&cursor[key], __popc(same));
    at = __shfl_sync(0xFFFFFFFFu, at, first);
    if (key >= 0) order[at + __popc(same & ((1u << lane) - 1u))] = p;
}

}  // namespace

cudaError_t launch_plan(const BatchView &b, const Scoring &sc, int32_t mode, const PlanBuffers &pb,
                        unsigned long long *need, cudaStream_t st) {
    cudaError_t e;
    if (b.npairs <= kPlanFew) {
        k_plan_small<3><<<1, kScanThreads, (kPlanBins >> 3) * 4, st>>>(b, sc, mode, pb, need);
        return cudaGetLastError();
    }
    if (b.npairs <= kPlanSmall) {
        static std::atomic<unsigned long long> ready{0};  // devices whose kernel has its shared-memory limit
        int dev = 0;
        if ((e = cudaGetDevice(&dev))) return e;
        if (dev >= 64 || !((ready.load() >> dev) & 1ull)) {
            if ((e = cudaFuncSetAttribute(k_plan_small<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPlanBins * 4)))
                return e;
            if (dev < 64) ready.fetch_or(1ull << dev);
        }
        k_plan_small<0><<<1, kScanThreads, kPlanBins * 4, st>>>(b, sc, mode, pb, need);
        return cudaGetLastError();
    }
    if ((e = cudaMemsetAsync(pb.hist, 0, sizeof(int32_t) * 2 * kPlanBins, st))) return e;
    const int nb = (b.npairs + 255) / 256;
    k_plan_keys<<<nb, 256, 0, st>>>(b, sc, mode, pb.keys, pb.hist);
    k_plan_scan<<<1, kScanThreads, 0, st>>>(pb.hist, pb.binoff, pb.var_start, pb.task_lo, pb.task_hi,
                                            pb.ntasks, pb.head);
    k_plan_scatter<<<nb, 256, 0, st>>>(b.npairs, pb.keys, pb.binoff, pb.cursor, pb.order);
    return cudaGetLastError();
}

bool plan_takes_needs(int npairs) { return npairs <= kPlanSmall; }
int plan_launches(int npairs) { return npairs <= kPlanSmall ? 1 : 3; }

}  // namespace gsw
