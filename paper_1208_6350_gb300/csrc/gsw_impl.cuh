// Internal declarations shared by the library's translation units (device
// kernels and the host runtime behind include/gsw.h).  Nothing here is part of
// the public ABI.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include <vector>

#include "gsw.h"

// Results owned by the library (gsw_align_batch_results, gsw_serve_poll_results):
// host copies of the records, the CIGAR words they index and, with GSW_COLMAX,
// the max arrays; released by gsw_results_free.
struct gsw_results {
    std::vector<gsw_result> res;
    std::vector<uint32_t> cigar;
    std::vector<int32_t> colmax;
    std::vector<int64_t> colmax_off;  // per pair, into colmax (empty without GSW_COLMAX)
    std::vector<int32_t> t_len;       // per pair
};

namespace gsw {

constexpr int kMaxAlpha = 32;

// Scoring scheme, passed by value to kernels (lives in the parameter bank).
struct Scoring {
    int32_t A;      // alphabet size
    int32_t O, X;   // gap open / extend, positive, O >= X: a gap of length k costs O + (k-1) X
    int32_t wmax;   // max matrix entry
    int32_t wmin;   // min matrix entry
    int32_t dna4;   // 1 when A == 4: the fill uses the letter-pair profile
    int32_t one;    // 1, unknown to the compiler: x * one + y issues as an integer multiply-add on the FMA pipe
    int8_t W[kMaxAlpha * kMaxAlpha];  // W[a * A + b]: query letter a vs target letter b
    // 16-bit fill class per query-row bucket: the tuned one, or the one
    // default_classes chose for the batch (-1: the smallest one-strip variant)
    int8_t fill_class[GSW_TUNE_BUCKETS];
    int8_t rev_class[GSW_TUNE_BUCKETS];  // of the reversed fill, + 1 (0: as the forward fill)
    // a pair whose strips one after the other take more steps runs on a CTA (0:
    // off), in the forward and in the reversed fill
    int32_t cta_steps, cta_steps_rev;
};

// Batch view (device pointers) shared by every stage.
struct BatchView {
    const uint8_t *q;
    const int64_t *q_off;
    const int32_t *q_len;
    const uint8_t *t;
    const int64_t *t_off;
    const int32_t *t_len;
    gsw_result *res;
    int32_t npairs;
    uint32_t flags;
    int32_t mask_len;  // < 0: max(m/2, 15)
    int32_t *colmax;
    const int64_t *colmax_off;
    uint32_t *cigar;
    int64_t cigar_cap;
    unsigned long long *cigar_cursor;
};

// Stage of the pipeline a fill launch serves.
enum FillMode : int32_t {
    kFillForward = 0,  // forward local fill: score1, ends, max array, secondary
    kFillRerun = 1,    // forward fill in 32-bit lanes for pairs whose 16-bit fill overflowed
    kFillReverse = 2,  // reversed fill from the end: begins (pairs whose reverse band is wide)
    kPlanBand = 3,     // not a fill: classes of the thread-per-pair band kernel
    kPlanTrace = 4,    // not a fill: pairs left to the warp traceback
};

// Kernel variants: (threads per pair P, row-words per thread R, 32-bit
// lanes).  A 16-bit variant covers 2*P*R query rows per strip, a 32-bit one
// P*R; longer queries run in several strips.  X(id, P, R, s32)
#define GSW_FILL_VARIANTS(X) \
    X(0, 16, 2, 0)           \
    X(1, 16, 3, 0)           \
    X(2, 16, 4, 0)           \
    X(3, 16, 5, 0)           \
    X(4, 16, 6, 0)           \
    X(5, 16, 7, 0)           \
    X(6, 16, 8, 0)           \
    X(7, 32, 8, 1)           \
    X(8, 8, 8, 0)            \
    X(9, 8, 10, 0)           \
    X(10, 8, 12, 0)          \
    X(11, 8, 14, 0)          \
    X(12, 8, 16, 0)          \
    X(13, 4, 6, 0)           \
    X(14, 4, 8, 0)           \
    X(15, 4, 10, 0)          \
    X(16, 4, 12, 0)          \
    X(17, 4, 14, 0)          \
    X(18, 4, 16, 0)          \
    X(19, 16, 10, 0)         \
    X(20, 16, 12, 0)         \
    X(21, 16, 16, 0)
struct Variant {
    int P, R, s32;
};
constexpr int kNumVariants = 22;
constexpr int kVarS32 = 7;
constexpr int kVarMaxS16 = 6;  // the tallest of 0..6, 16 lanes and 2..8 row words
// 8..12: one pair per 8 lanes with 8..16 row words per lane (128..256 rows per
// strip): twice the cells per lane and step of the 16-lane variants, so the
// per-step costs (shuffles, letter loads, trackers) weigh half as much; taken
// by large batches (default_classes) and by tune tables
constexpr int kVarP8First = 8;
// 13..18: one pair per 4 lanes with 6..16 row words per lane (48..128 rows per
// strip): half the wavefront's skew again and strips that fit reads of up to
// 128 rows closely; 4-letter alphabets only (a general alphabet's profile
// would leave few warps per SM)
constexpr int kVarP4First = 13;
// 19..21: one pair per 16 lanes with 10, 12 or 16 row words per lane (320, 384
// or 512 rows per strip): queries of 257 to 512 rows in one strip, without the
// boundary rows and the second pass over the target
constexpr int kVarTallFirst = 19;
__host__ __device__ constexpr bool is_p8(int v) { return v >= kVarP8First && v < kVarP4First; }
__host__ __device__ constexpr bool is_p4(int v) { return v >= kVarP4First && v < kVarTallFirst; }
// Two more fill classes: pairs whose query spans many strips run on a whole
// CTA (k_fill_long), one 32-lane warp per strip, strips pipelined across the
// CTA's warps; 16-bit lanes (2*32*16 = 1,024 rows per strip for DNA, 2*32*8 =
// 512 for general alphabets) or 32-bit lanes (256 rows per strip).  One pair
// per task.
constexpr int kClassLong16 = kNumVariants;
constexpr int kClassLong32 = kNumVariants + 1;
constexpr int kNumFillClasses = kNumVariants + 2;
__host__ __device__ inline Variant variant_at(int v) {
    switch (v) {
#define GSW_VARIANT_CASE(id, P, R, S32) \
    case id: return Variant{P, R, S32};
        GSW_FILL_VARIANTS(GSW_VARIANT_CASE)
#undef GSW_VARIANT_CASE
    case kClassLong16: return Variant{32, 16, 0};  // (DNA; general alphabets 8 row words)
    default: return Variant{32, 8, 1};
    }
}
// A query goes to the CTA kernel when it spans more than 3.5 x 512 rows of
// 4-letter DNA (a few such pairs in flight keep every warp busy), or more than
// 8 x 512 rows of a general alphabet (whose CTA holds fewer warps per SM).
__host__ __device__ inline bool long_pair(int rows, bool s32, bool dna) {
    const int sp = s32 ? 256 : 512;
    return dna ? 2 * rows > 7 * sp : rows > 8 * sp;
}
__host__ __device__ inline int variant_rows(int v) {
    Variant x = variant_at(v);
    return x.s32 ? x.P * x.R : 2 * x.P * x.R;
}

// The smallest one-strip 16-lane variant holding a query of `rows`, or the
// tallest (several strips).
__host__ __device__ inline int pick_s16(int rows) {
    for (int v = 0; v <= kVarMaxS16; v++)
        if (variant_rows(v) >= rows) return v;
    return kVarMaxS16;
}

// What a tune table gives bucket b: the class it names, or the default rule (-1)
// where it holds rates (gsw_autotune's do) and the default rule's is no lower.
inline int tuned_class(const gsw_tune &t, int b) {
    return t.gcups_default[b] > 0 && t.gcups_default[b] >= t.gcups[b] ? -1 : t.fill_class[b];
}

// 16-bit fill class of a query of `rows` (>= 1): the tuned class of its
// bucket, else the smallest one-strip variant, or the CTA class for queries
// of many strips.
__host__ __device__ inline int pick_class16(int rows, const Scoring &sc) {
    const int b = (rows - 1) / GSW_TUNE_ROWS;
    if (rows >= 1 && b < GSW_TUNE_BUCKETS && sc.fill_class[b] >= 0) {
        const int c = sc.fill_class[b];  // public codes: 0..6, 8 CTA, 9..13 8-lane variants
        return c == 8 ? kClassLong16 : (c >= 9 ? kVarP8First + (c - 9) : c);
    }
    return long_pair(rows, false, sc.dna4) ? kClassLong16 : pick_s16(rows);
}

// Class of the reversed fill of a query whose end row is rows - 1 (plan.cu):
// the forward rule, or the 32-bit classes for a pair in 32-bit lanes; a DNA
// query of several strips reverses in the CTA kernel.
__host__ __device__ inline int pick_class_reverse(int rows, bool s32, const Scoring &sc) {
    const int b = (rows - 1) / GSW_TUNE_ROWS;
    int v;
    if (s32) v = long_pair(rows, true, sc.dna4) ? kClassLong32 : kVarS32;
    else if (rows >= 1 && b < GSW_TUNE_BUCKETS && sc.rev_class[b] > 0) v = sc.rev_class[b] - 1;
    else v = pick_class16(rows, sc);
    if (sc.dna4 && v != kClassLong16 && v != kClassLong32 && rows > variant_rows(v))
        v = v == kVarS32 ? kClassLong32 : kClassLong16;
    return v;
}

// A pair of at most rows x cols letters cannot leave the lanes whose clamp is
// a half-precision multiply-add (fill.cuh, LH): a local score is at most
// min(rows, cols) x the largest matrix entry, and every lane value at most the
// score + O + one matrix entry, which must stay within the integers half
// precision holds exactly (2048); O >= -wmin keeps the sums of the shifted
// scores non-negative (signed bytes outside the 4-letter alphabets).
__host__ __device__ inline bool half_fits(int rows, int cols, const Scoring &sc) {
    if (sc.O < -sc.wmin || (!sc.dna4 && sc.wmax + sc.O > 127)) return false;
    const long long top = sc.wmax > 0 ? sc.wmax : 0;
    return (rows < cols ? rows : cols) * top + top + sc.O <= 2047;
}

// Whether a tune table names the class of queries of `rows` (the default rule
// marks the buckets it fills in by their rev_class).
__host__ __device__ inline bool tuned_rows(int rows, const Scoring &sc) {
    const int b = (rows - 1) / GSW_TUNE_ROWS;
    return rows >= 1 && b < GSW_TUNE_BUCKETS && sc.fill_class[b] >= 0 && sc.rev_class[b] == 0;
}

// Whether a pair that class v would run strip after strip goes to the CTA
// class instead (sc.cta_steps, default_classes).  Not where a tune table names
// the class: there its strips run one after the other as the table says.
__host__ __device__ inline bool cta_pair(int v, int rows, int cols, const Scoring &sc, bool reverse) {
    const int32_t most = reverse ? sc.cta_steps_rev : sc.cta_steps;
    if (most <= 0 || v >= kNumVariants || v == kVarS32 || tuned_rows(rows, sc)) return false;
    const int strips = (rows + variant_rows(v) - 1) / variant_rows(v);
    // (a step's time grows with its row words; 0.3 us is that of 8)
    return strips > 1 && (long long)strips * cols * (4 + variant_at(v).R) > 12LL * most;
}

// A batch whose pairs have on average at least a quarter of the largest one's
// cells.
inline bool even_batch(int npairs, int maxm, int maxn, double cells) {
    return cells >= 0.25 * npairs * (double)maxm * maxn;
}
// ... of pairs that are nearly alike: at least three quarters
inline bool equal_batch(int npairs, int maxm, int maxn, double cells) {
    return cells >= 0.75 * npairs * (double)maxm * maxn;
}

// Chooses the fill classes of a batch's untuned buckets from its size (pairs,
// longest target, forward cells).
//
// A class costs its strips x the time of a strip's step.  The table holds that
// time (ps per pair and column on a whole GB300, measured with the chip full:
// 6 G cells of equal pairs, targets of 650 letters, 360 for 20-letter
// alphabets); strips of a query that needs several cost kMulti times as much
// (boundary rows in and out).  Narrower groups pay less skew and fewer per-step
// instructions per pair but need more pairs to fill the chip: 8 lanes from
// 8,192 pairs (100 rows, 1,000 columns: 883 GCUPS against 1,155 at 3,000 pairs,
// 2,503 against 2,307 at 10,000), 4 lanes from 16,384 (1,888 against 2,503 at
// 10,000 pairs, 3,907 against 3,193 at 92,000).  A pair of several strips that
// alone would take more than about a quarter of the batch's time (its steps x 0.3 us
// against the cells at 2.5 T cells/s; 0.46 us and 1.5 T for general alphabets)
// runs its strips side by side on a CTA (600 x 1,000 DNA: 1,851 GCUPS against
// 1,513 at 3,000 pairs; 350 x 360 protein: 691 against 330 at 1,000 pairs).
//
// Not in an even batch (even_batch) of more pairs than the 16-lane groups that
// can be resident, kWave: there no pair outlives the others, and a part of them
// on CTAs, where strips wait for each other, only takes SMs from the groups
// (750-1,500 x 600-1,200 DNA: 4,000 pairs 2.53 ms with CTAs, 3.05 without; 6,000 pairs 3.52 and 3.09;
// 10,000 pairs 5.07 and 4.28).  For general alphabets from half as many pairs on,
// where queries have at most 1,024 rows: two CTA strips, which leave half of a
// CTA's warps idle (450-900 x 400-800 protein: 1,000 pairs 0.57 ms with CTAs,
// 1.42 without; 4,000 pairs 1.55 and 1.22; 10,000 pairs 2.68 and 3.03, so from
// kWide pairs on only up to 768 rows: 300-600 x 200-400 1.45 and 0.93).
//
// General alphabets in less than kWave pairs: a class costs its pairs' latency,
// strips x the row words of a step, not its share of a full chip (225-450 x
// 200-400: 2,500 pairs 0.490 -> 0.355 ms, 300-600 x 200-400: 4,000 pairs 0.768
// -> 0.583 ms, with the rule above), where CTAs do not take the tall ones.
//
// Both forward only: reversed pairs end at their begins, unlike each other (3,000
// pairs of 350-700 x 200-400 protein with CIGARs 2.06 ms, with both rules in the
// reversed fill too 2.59).
inline void default_classes(Scoring &sc, int npairs, int maxm, int maxn, double cells) {
    constexpr int kWide = 8192, kNarrow = 16384, kFewPairs = 2048;
    constexpr int kWave = 152 * 4 * 8;  // SMs x blocks of 4 warps x pairs of a block
    // (a power of two: batches of like size keep their captured graphs)
    sc.cta_steps = 256;
    while (sc.cta_steps < cells * 3.5e-7 && sc.cta_steps < (1 << 28)) sc.cta_steps *= 2;
    sc.cta_steps_rev = sc.cta_steps;
    const bool even = even_batch(npairs, maxm, maxn, cells);
    if (even && (sc.dna4 ? npairs > kWave : npairs > kWave / 2 && maxm <= (npairs > kWide ? 768 : 1024))) sc.cta_steps = 0;
    static constexpr float dna[kNumVariants] = {28.3f, 33.4f, 39.2f, 45.8f, 50.1f, 59.6f, 61.2f, 0,
                                                32.1f, 36.3f, 42.6f, 52.3f, 55.8f, 13.8f, 16.8f, 19.5f,
                                                21.4f, 24.8f, 29.5f, 72.6f, 85.0f, 112.0f};
    static constexpr float gen[kNumVariants] = {32.0f, 41.5f, 47.4f, 57.7f, 65.0f, 84.2f, 94.9f, 0,
                                                39.7f, 48.0f, 59.5f, 73.7f, 97.1f, 0,     0,     0,
                                                0,     0,     0,     110.0f, 136.0f, 203.0f};
    for (int b = 0; b < GSW_TUNE_BUCKETS; b++) {
        if (sc.fill_class[b] >= 0) continue;
        const int rows = (b + 1) * GSW_TUNE_ROWS;
        if (long_pair(rows, false, sc.dna4)) continue;
        const float multi = sc.dna4 ? 1.3f : 1.08f;
        const bool latency = !sc.dna4 && npairs < kWave && (sc.cta_steps == 0 || rows <= 512);
        float best = 0, best16 = 0;
        int pick = -1, pick16 = -1;
        for (int v = 0; v < kNumVariants; v++) {
            const bool p8 = is_p8(v), p4 = is_p4(v);
            if (v == kVarS32) continue;
            if (p8 && (npairs < kWide || rows > variant_rows(v))) continue;
            if (p4 && (npairs < kNarrow || rows > variant_rows(v) || !sc.dna4 || !half_fits(rows, maxn, sc))) continue;
            const int strips = (rows + variant_rows(v) - 1) / variant_rows(v);
            const float full = strips * (sc.dna4 ? dna[v] : gen[v]) * (strips > 1 ? multi : 1.0f);
            const float cost = latency ? (float)strips * (4 + variant_at(v).R) : full;
            if (pick < 0 || cost < best) {
                best = cost;
                pick = v;
            }
            if (!p8 && !p4 && (pick16 < 0 || full < best16)) {
                best16 = full;
                pick16 = v;
            }
        }
        // (codes of the table, pick_class16)
        sc.fill_class[b] = (int8_t)(pick >= kVarP8First ? 9 + (pick - kVarP8First) : pick);
        sc.rev_class[b] = (int8_t)(pick16 + 1);
    }
    // a batch that leaves the chip half empty reverses every query (of one strip)
    // in the longest one's class: one launch instead of one per class below it,
    // and its time is the longest pair's anyway
    const int top = maxm < 1 ? 0 : (maxm - 1) / GSW_TUNE_ROWS;
    if (npairs < kFewPairs && top < GSW_TUNE_BUCKETS && sc.rev_class[top] > 0 && variant_rows(sc.rev_class[top] - 1) >= maxm)
        for (int b = 0; b < top; b++)
            if (sc.rev_class[b] > 0) sc.rev_class[b] = sc.rev_class[top];
}

// The fill classes a launch of `mode` can meet when every query has minm to
// maxm rows (a superset; each fill launch leaves the other classes out; the
// reversed fill's queries end anywhere, so have 1 to maxm).
// force_s32: the batch runs in 32-bit lanes; s32: some pair may have been
// refilled in 32-bit lanes.  Empty pairs of the forward fill take class 0.
inline uint32_t fill_class_mask(int mode, int maxm, const Scoring &sc, bool force_s32, bool s32,
                                int minm = 0) {
    uint32_t m = 0;
    const int upto = maxm < GSW_TUNE_BUCKETS * GSW_TUNE_ROWS ? maxm : GSW_TUNE_BUCKETS * GSW_TUNE_ROWS;
    if (mode == kFillForward && force_s32) return (1u << kVarS32) | (1u << kClassLong32);
    if (mode == kFillRerun) return (1u << kVarS32) | (1u << kClassLong32);
    if (mode == kFillForward && minm <= 0) m |= 1u << 0;
    bool strips = maxm > upto;  // some class of the default rule can hold a pair of several strips
    for (int r = 1; r <= upto; r++) {
        if (mode == kFillForward && r < minm) continue;
        const int c = mode == kFillForward ? pick_class16(r, sc) : pick_class_reverse(r, false, sc);
        m |= 1u << c;
        strips |= r > variant_rows(c) && !tuned_rows(r, sc);
        if (s32 && mode != kFillForward) m |= 1u << pick_class_reverse(r, true, sc);
    }
    if ((mode == kFillForward ? sc.cta_steps : sc.cta_steps_rev) > 0 && strips) m |= 1u << kClassLong16;
    if (maxm > upto) {  // past the tuned buckets: the tallest variant or the CTA classes
        m |= (1u << kVarMaxS16) | (1u << kClassLong16);
        if (s32 && mode != kFillForward) m |= (1u << kVarS32) | (1u << kClassLong32);
    }
    return m;
}

// Most rows a class of a launch can hold when no query has more than maxm.
struct ClassRows {
    int most[kNumFillClasses] = {};
};
inline ClassRows fill_class_rows(int mode, int maxm, const Scoring &sc, uint32_t mask) {
    ClassRows r;
    const int upto = maxm < GSW_TUNE_BUCKETS * GSW_TUNE_ROWS ? maxm : GSW_TUNE_BUCKETS * GSW_TUNE_ROWS;
    for (int x = 1; x <= upto; x++)
        r.most[mode == kFillForward ? pick_class16(x, sc) : pick_class_reverse(x, false, sc)] = x;
    if (maxm > upto) r.most[kVarMaxS16] = maxm;
    for (int c : {kVarS32, kClassLong16, kClassLong32}) r.most[c] = maxm;
    for (int c = 0; c < kNumFillClasses; c++)
        if (!((mask >> c) & 1u)) r.most[c] = 0;
    return r;
}

// The classes of a launch whose pairs all fit the half-precision clamp lanes.
inline uint32_t fill_half_mask(const ClassRows &rows, int maxn, const Scoring &sc) {
    uint32_t m = 0;
    for (int c = 0; c < kNumVariants; c++)
        if (!variant_at(c).s32 && half_fits(rows.most[c], maxn, sc)) m |= 1u << c;
    return m;
}

// The classes that can hold a pair of several strips (which needs boundary rows).
inline uint32_t fill_multi_mask(const ClassRows &rows) {
    uint32_t m = (1u << kClassLong16) | (1u << kClassLong32);
    for (int c = 0; c < kNumVariants; c++)
        if (rows.most[c] > variant_rows(c)) m |= 1u << c;
    return m;
}

// Work plan of one fill launch: pairs sorted by (variant, cost descending),
// cut into warp tasks of 32/P pairs of one variant.  Task indices are handed
// out heaviest variant first (variant index descending).
struct FillPlan {
    const int32_t *order;      // sorted pair indices
    const int32_t *var_start;  // [kNumFillClasses+1] start of each class's pairs in `order`
    const int32_t *task_lo;    // [kNumFillClasses] first task index of each class
    const int32_t *task_hi;    // [kNumFillClasses] one past its last task index
    int32_t *head;             // [kNumFillClasses] task counters (zeroed by the plan)
    const int32_t *ntasks;     // total tasks
};

// Scratch of the fill launches: each launch (they run one after the other)
// lays out its own slots, one per pair in flight (column maxima, then boundary
// rows), as wide as its lanes need.
struct FillScratch {
    void *base;
    size_t bytes;
    size_t bnd_off;  // the launch's boundary rows start here
    int32_t ncap;    // columns per slot (a multiple of 4: 8-byte stores of four 16-bit maxima)
};

// CTAs that share the pairs of a launch of the CTA kernels: as many as a pair's
// strips fill (`want`, a power of two up to `most`) where the batch's few pairs
// leave the chip to the longest one, else one.  One also where other batches
// need the chip meanwhile (one_cta: a server's heavy worker): a cluster's CTAs hold
// their SMs until its longest pair ends, most of them waiting at its barriers
// (mixed stream at 10,000 requests/s: 1,193 GCUPS with clusters, 1,254 without).
inline int cluster_ctas(int npairs, int few, int want, int most, bool one_cta) {
    int c = 1;
    if (npairs <= few && !one_cta)
        while (c < want && c < most) c *= 2;
    return c;
}

// The same for a batch of like pairs (equal_batch) of `strips` each: the CTAs a
// cluster, up to the c above, with which the resident CTAs' warps run their pairs'
// strips in the fewest rounds, or the fewest CTAs (300 pairs of 4,500 x 4,000 on
// 456 CTAs: 3.60 ms in clusters of 2, 2.75 without; 500 pairs: 4.13 and 5.57).
inline int cluster_ctas_alike(int npairs, int strips, int warps, int resident, int c) {
    int best = 1, fewest = 0;
    for (int x = 1; x <= c; x *= 2) {
        const int clusters = resident / x > 0 ? resident / x : 1;
        const int pairs = (npairs + clusters - 1) / clusters;  // of a cluster
        const int rounds = (pairs * strips + warps * x - 1) / (warps * x);
        if (x == 1 || rounds < fewest) {
            fewest = rounds;
            best = x;
        }
    }
    return best;
}

struct FillLaunch {
    BatchView b;
    Scoring sc;
    FillPlan plan;
    FillScratch scr;
    int32_t mode;
    int32_t maxm;         // longest query
    bool one_cta;         // no clusters (cluster_ctas)
    bool equal;           // equal_batch
    uint32_t class_mask;  // classes launched (bit c: class c); the others hold no pair
    uint32_t multi_mask;  // classes that can hold pairs of several strips
    uint32_t half_mask;   // classes whose values stay below 2048: the half-precision clamp lanes
    // nonzero once the batch's letter check found a code >= the alphabet
    // (written by the check, which runs first on the stream): the fill then
    // writes empty records and touches no letter, so its steady steps need
    // no clamp (the call returns GSW_EINVAL)
    const int32_t *bad_letters;
};

// internal per-pair bits (besides the public GSW_RES_*)
constexpr int32_t kResPendingS32 = 0x40;  // 16-bit fill overflowed: refill in 32-bit lanes
constexpr int32_t kResInternal = GSW_RES_INTERNAL;  // a consistency check failed (should never happen)
constexpr int32_t kResInvalid = GSW_RES_INVALID;    // gsw_fill_static: the pair's inputs were rejected
constexpr int32_t kResPendingTrace = 0x100;  // band too wide for one thread: warp traceback

// The thread-per-pair band kernel handles bands up to this many diagonals and
// this many rows; wider or longer pairs use the ring reverse fill and the warp
// traceback.
constexpr int kBandMaxWidth = 32;
constexpr int kBandMaxRows = 4096;
// Reverse bands the thread-per-pair kernel takes; wider ones reverse in the
// 16-bit ring fill (the begin), the CIGAR still comes from the band kernel
// when the traceback band is narrow.  (Measured with 16 on the short-read
// workload: band 8.26 -> 6.69 ms but ring reverse 1.89 -> 3.99 ms, so 32.)
constexpr int kBandMaxRevWidth = 32;

// Below this many pairs the thread-per-pair band kernel would occupy a few
// percent of the GPU's threads: the begins then come from the ring reverse
// fill and the CIGARs from the warp tracebacks.
constexpr int kSmallBatch = 1 << 14;
__host__ __device__ inline bool small_batch(const BatchView &b) { return b.npairs < kSmallBatch; }

constexpr int kPlanBinsPerVariant = 1024;
constexpr int kPlanBins = kNumFillClasses * kPlanBinsPerVariant;

// Width of the window the reversed fill scans, ending at the end column: an
// optimal alignment ending at (end_q, end_t) with score1 has at most
// D = ((end_q+1)*wmax - score1 - O)/X + 1 target letters against gaps (every
// gap run costs at least O + (len-1)X when O >= X), so it begins within
// end_q + 1 + D columns of the end.
__host__ __device__ inline int reverse_window(int end_q, int end_t, int score1, const Scoring &sc) {
    if (sc.X <= 0) return end_t + 1;
    long long d = (long long)(end_q + 1) * sc.wmax - score1 - sc.O;
    d = d < 0 ? 0 : d / sc.X + 1;
    long long w = (long long)end_q + 1 + d;
    long long lim = (long long)end_t + 1;
    return (int)(w < lim ? w : lim);
}

// Largest number of gap letters an alignment ending at (end_q, end_t) with
// score1 can hold: its at most end_q+1 aligned pairs score <= (end_q+1)*wmax,
// and g gap letters cost at least O + (g-1)X (O >= X).  -1 means unbounded.
__host__ __device__ inline int reverse_gap_bound(int end_q, int score1, const Scoring &sc) {
    long long num = (long long)(end_q + 1) * sc.wmax - score1 - sc.O;
    if (num < 0) return 0;
    if (sc.X <= 0) return -1;
    long long g = num / sc.X + 1;
    return g > (1 << 30) ? (1 << 30) : (int)g;
}

// Largest number of query letters against gaps it can hold: each also takes
// a row from the at most end_q+1 that could be aligned pairs, so g of them
// satisfy (end_q+1-g)*wmax - O - (g-1)X >= score1.  On the reversed
// sequences these are the steps below the main diagonal: the reverse band is
// [-reverse_gap_bound_rows, reverse_gap_bound], much narrower below.
__host__ __device__ inline int reverse_gap_bound_rows(int end_q, int score1, const Scoring &sc) {
    const long long num = (long long)(end_q + 1) * sc.wmax - score1 - sc.O + sc.X;
    const long long den = (long long)sc.wmax + sc.X;
    if (num < 0 || den <= 0) return 0;
    const long long g = num / den;
    return g > end_q + 1 ? end_q + 1 : (int)g;
}

// Diagonals of the reverse band: G above, reverse_gap_bound_rows below; -1
// when unbounded (extend 0)
__host__ __device__ inline int reverse_band_width(int end_q, int score1, const Scoring &sc) {
    const int G = reverse_gap_bound(end_q, score1, sc);
    if (G < 0) return -1;
    return G + reverse_gap_bound_rows(end_q, score1, sc) + 1;
}

// Half-width of the band of the global alignment between begin and end
// (la x lb letters, optimum score1): a path through diagonal d has at least
// g = |d| + |lb - la - d| gap letters and (la + lb - g)/2 aligned pairs, so
// scores at most wmax*floor((la+lb-g)/2) - O - (g-1)X; diagonals where that
// bound is below score1 carry no optimal path.  Returns w such that the band
// is [min(0, lb-la) - w, max(0, lb-la) + w].
__host__ __device__ inline int band_halfwidth(int la, int lb, int score1, const Scoring &sc) {
    const int delta = lb - la;
    const int g0 = delta < 0 ? -delta : delta;
    auto ub = [&](long long g) -> long long {
        long long aligned = ((long long)la + lb - g) / 2;
        long long s = (long long)sc.wmax * aligned;
        if (g > 0) s -= sc.O + (g - 1) * (long long)sc.X;
        return s;
    };
    // largest w with ub(g0 + 2w) >= score1 (ub is non-increasing in g)
    int lo = 0, hi = la + lb + 1;
    while (lo < hi) {
        int mid = (lo + hi + 1) / 2;
        if (ub(g0 + 2LL * mid) >= score1) lo = mid;
        else hi = mid - 1;
    }
    return lo;
}

// Diagonal range [dlo, dhi] of the traceback band, clipped to the rectangle.
__host__ __device__ inline int band_range(int la, int lb, int score1, const Scoring &sc, int *dlo, int *dhi) {
    const int w = band_halfwidth(la, lb, score1, sc);
    const int delta = lb - la;
    int lo = (delta < 0 ? delta : 0) - w, hi = (delta > 0 ? delta : 0) + w;
    lo = lo < -la ? -la : lo;
    hi = hi > lb ? lb : hi;
    *dlo = lo;
    *dhi = hi;
    return hi - lo + 1;
}

// Traceback classes of the pairs the band kernel leaves (bands wider than 32
// diagonals, or small batches): 0-3 anti-diagonal warp kernel (bands of at
// most 64/128/256/512 diagonals), 4 the CTA strip kernel (wider bands), 5-8
// the 16-bit full-rectangle kernel.  DNA: 5-8, strips of 64/128/192/256 query
// rows (8 lanes x R = 4/8/12/16 words x 2 halves; taller regions run several
// 256-row strips).  Other alphabets: 5, and 6 with a larger scratch allowance
// for regions whose scratch would exceed kT16MaxWords (strips by t16_shape).
constexpr int kTraceRingClass = 4;
constexpr int kTraceT16First = 5;
constexpr int kTraceT16Classes = 4;
constexpr int kT16P = 8;                   // lanes per pair
constexpr int kT16MaxCols = 4096;          // longest target region of the 16-bit kernel
constexpr long long kT16MaxWords = 1 << 17;  // scratch words of one pair (512 KB), as launched
// general alphabets: regions over kT16MaxWords take class 6 with this
// allowance (its own launch and scratch, so the few large pairs do not shrink
// the groups of the others)
constexpr long long kT16MaxWordsBig = 1 << 20;
// 8 lanes and strips of 64(v+1) rows: the shapes of DNA's classes v, and of
// v = 0 for other alphabets
__host__ __device__ inline int t16_R(int v) { return 4 * (v + 1); }
__host__ __device__ inline int t16_strip_rows(int v) { return 2 * kT16P * t16_R(v); }
__host__ __device__ inline int t16_strips(int la, int v) { return (la + t16_strip_rows(v) - 1) / t16_strip_rows(v); }
__host__ __device__ inline int t16_steps(int lb) { return lb + 2 * kT16P - 1; }
// direction words of one pair (strips x steps x R/4 words x 8 lanes)
__host__ __device__ inline long long t16_dir_words(int la, int lb, int v) {
    return (long long)t16_strips(la, v) * t16_steps(lb) * (t16_R(v) / 4) * kT16P;
}
// scratch words of one pair: direction words, then two boundary rows (one
// word per column) when it has several strips
__host__ __device__ inline long long t16_need_words(int la, int lb, int v) {
    const long long d = t16_dir_words(la, lb, v);
    return t16_strips(la, v) > 1 ? d + 2LL * ((lb + 3) & ~3) : d;
}
// How launch class v runs: P lanes a pair and R row words a lane, so strips of
// 2PR rows.  DNA: the trace class's.  Other alphabets have three launches: v = 0
// (64-row strips), and whole warps with 256-row strips for v = 1 (regions over
// kT16MaxWords) and v = 2 (regions of trace class 5 taller than kT16Tall
// rows): a group of 8 lanes runs the 16 strips of a 1,000-row
// region one after the other, and beside the bulk of the pairs those few
// regions then ended last (40 x 1,000 protein pairs: traceback 9.0 -> 5.9 ms).
struct T16Shape {
    int P, R;
    __host__ __device__ int rows() const { return 2 * P * R; }
    __host__ __device__ int strips(int la) const { return (la + rows() - 1) / rows(); }
    __host__ __device__ int steps(int lb) const { return lb + 2 * P - 1; }
    __host__ __device__ long long need_words(int la, int lb) const {
        const long long d = (long long)strips(la) * steps(lb) * (R / 4) * P;
        return strips(la) > 1 ? d + 2LL * ((lb + 3) & ~3) : d;
    }
};
constexpr int kT16Tall = 256;
__host__ __device__ inline T16Shape t16_shape(int v, bool dna) {
    return dna ? T16Shape{kT16P, t16_R(v)} : (v == 0 ? T16Shape{kT16P, 4} : T16Shape{32, 4});
}
// launch class of a region trace_class gave class c
__host__ __device__ inline int t16_launch_class(int c, int la, bool dna) {
    return !dna && c == kTraceT16First && la > kT16Tall ? kTraceT16First + 2 : c;
}
// small: a batch of fewer than 2^14 pairs (the rectangle needs a wider margin
// there, where the anti-diagonal kernel's one pair per warp keeps more pairs
// in flight)
__host__ __device__ inline int trace_class(int la, int lb, int score1, const Scoring &sc, bool small, int *dlo,
                                           int *dhi) {
    const int width = band_range(la, lb, score1, sc, dlo, dhi);
    const int ad = width <= 64 ? 0 : width <= 128 ? 1 : width <= 256 ? 2 : width <= 512 ? 3 : kTraceRingClass;
    if (la >= 1 && lb >= 1 && lb <= kT16MaxCols) {
        // the shape of the launch the region would take; general alphabets keep
        // A x R profile words per lane, so their 8-lane strips have 64 rows (128
        // measured 2.5 % slower on protein search: a third of the warps per SM)
        const bool dna = sc.dna4 != 0;
        int v = dna ? (la - 1) / 64 : 0;
        v = v < kTraceT16Classes ? v : kTraceT16Classes - 1;
        T16Shape shape = t16_shape(t16_launch_class(kTraceT16First + v, la, dna) - kTraceT16First, dna);
        long long cap = kT16MaxWords;
        if (!dna && shape.need_words(la, lb) > kT16MaxWords) {
            v = 1;
            shape = t16_shape(v, dna);
            cap = kT16MaxWordsBig;
        }
        const long long rows = (long long)shape.strips(la) * shape.rows();
        const long long cols = lb + 2 * shape.P;
        // every value of the DP over the padded rectangle lies in
        // [-(3O + X(rows + cols) + |wmin|), wmax * min(rows, cols) + wmax]:
        // it must fit a biased 16-bit lane
        const long long lo = 3LL * sc.O + (long long)sc.X * (rows + cols + 2) - (sc.wmin < 0 ? sc.wmin : 0);
        const long long hi = (long long)sc.wmax * ((cols < rows ? cols : rows) + 1);
        if (lo <= 30000 && hi <= 30000 && shape.need_words(la, lb) <= cap) {
            // cell updates: the rectangle, in 8-lane strips whatever shape runs
            // it, against the band's anti-diagonal slots; a 16-bit pair of cells
            // costs about the instructions of one 32-bit anti-diagonal cell (whole
            // warps' own padding counts for less: costed by it, too many regions of
            // general alphabets took the anti-diagonals, 1,000 calls' pairs of
            // 750-1,500 x 750-1,500 with CIGARs 5.1 -> 7.1 ms)
            // (bands wider than 512 diagonals: the rectangle always)
            const long long rect = (long long)t16_strips(la, v) * t16_strip_rows(v) * t16_steps(lb);
            if (ad == kTraceRingClass) return kTraceT16First + v;
            const long long band = (32LL << ad) * (la + lb + 1);
            if (rect <= (small ? 2 : 3) * band) return kTraceT16First + v;
        }
    }
    return ad;
}

// decision words of one pair in the anti-diagonal kernel: 8 anti-diagonals per
// word row, nch x 32 words a row
__host__ __device__ inline long long ad_dir_words(int la, int lb, int nch) {
    return ((long long)(la + lb + 1 + 7) / 8) * nch * 32;
}

// pairs left to the warp tracebacks
__host__ __device__ inline bool wants_trace(const gsw_result &r) {
    return r.score1 > 0 && (r.flags & kResPendingTrace) && !(r.flags & kResInternal) && r.read_begin1 >= 0 &&
           r.ref_begin1 >= 0;
}

// Largest needs of the warp tracebacks' pairs: [0] direction words of the
// anti-diagonal classes, [1] op words (anti-diagonal and 16-bit classes),
// [2..4] wide bands (launch_ring_needs: total words, largest pair, largest op
// words), [5] bit c: anti-diagonal class c has pairs, [6 + v] direction words of
// 16-bit launch class v (per group)
constexpr int kNeedMask = 5, kNeed16 = 6, kNeedWords = kNeed16 + kTraceT16Classes;
// A pair's share of those (v zeroed by the caller; the ring words are not set).
__host__ __device__ inline void trace_needs(const gsw_result &r, const Scoring &sc, bool small, unsigned v[kNeedWords]) {
    if (!wants_trace(r)) return;
    const int la = r.read_end1 - r.read_begin1 + 1, lb = r.ref_end1 - r.ref_begin1 + 1;
    const long long top = 0xFFFFFFFFLL;
    auto capped = [&](long long x) { return (unsigned)(x < top ? x : top); };
    int dlo, dhi;
    const int cls = trace_class(la, lb, r.score1, sc, small, &dlo, &dhi);
    if (cls == kTraceRingClass) return;
    v[1] = capped((long long)la + lb + 2);
    if (cls < kTraceRingClass) {
        v[0] = capped(ad_dir_words(la, lb, 1 << cls));
        v[kNeedMask] = 1u << cls;
    } else {
        const int c = t16_launch_class(cls, la, sc.dna4 != 0) - kTraceT16First;
        v[kNeed16 + c] = capped(t16_shape(c, sc.dna4 != 0).need_words(la, lb));
    }
}

// Whether a pair of a batch with these largest lengths can be of the wide-band
// class: not when every region the lengths allow fits the anti-diagonal kernel
// (at most 512 diagonals) or the 16-bit rectangle (trace_class; its needs and
// value ranges grow with the lengths).
inline bool ring_possible(int maxm, int maxn, const Scoring &sc) {
    if (maxm + maxn + 1 <= 512) return false;
    if (maxn > kT16MaxCols) return true;
    const long long rows = (long long)maxm + 256, cols = maxn + 2 * (sc.dna4 ? kT16P : 32);
    const long long lo = 3LL * sc.O + (long long)sc.X * (rows + cols + 2) - (sc.wmin < 0 ? sc.wmin : 0);
    const long long hi = (long long)sc.wmax * ((cols < rows ? cols : rows) + 1);
    if (lo > 30000 || hi > 30000) return true;
    const int m = maxm < 1 ? 1 : maxm, n = maxn < 1 ? 1 : maxn;
    if (sc.dna4) return t16_need_words(m, n, kTraceT16Classes - 1) > kT16MaxWords;
    return t16_shape(1, false).need_words(m, n) > kT16MaxWordsBig;
}

#ifdef __CUDACC__
// Row 2w + odd of byte-profile words lo (the low letter's) and hi (the high
// letter's): the low half's score of lo and the high half's of hi, sign-extended
__device__ __forceinline__ uint32_t merge_bytes(uint32_t lo, uint32_t hi, int odd) {
    uint32_t r;
    if (odd) asm("prmt.b32 %0, %1, %2, 0xF7A2;" : "=r"(r) : "r"(lo), "r"(hi));
    else asm("prmt.b32 %0, %1, %2, 0xD580;" : "=r"(r) : "r"(lo), "r"(hi));
    return r;
}
#endif

// stage launchers (host side, enqueue on `st`)
// Status of a completed batch from what its kernels counted, in order of
// precedence: letter codes outside the alphabet (GSW_EINVAL), records that
// failed a consistency check (GSW_EINTERNAL), CIGAR words beyond the
// caller's capacity (GSW_ECIGAR_SPACE, only with GSW_CIGAR).
__host__ __device__ inline int batch_status(int bad_letters, unsigned long long internal, bool cigar,
                                            unsigned long long cigar_words, long long cigar_capacity) {
    if (bad_letters) return GSW_EINVAL;
    if (internal) return GSW_EINTERNAL;
    if (cigar && cigar_words > (unsigned long long)(cigar_capacity < 0 ? 0 : cigar_capacity)) return GSW_ECIGAR_SPACE;
    return GSW_OK;
}

// Host helpers of the runtime (api.cu): the calling thread's error detail,
// the scoring checks shared by every entry point, and the count of records
// flagged kResInternal (one small kernel and a readback on `st`).
int set_err(int code, const char *fmt, ...);
int make_scoring(const int8_t *matrix, int32_t A, int32_t O, int32_t X, Scoring *sc);
cudaError_t launch_count_flag(const gsw_result *res, int32_t n, int32_t flag, unsigned long long *count,
                              cudaStream_t st);

// A record whose begins were asked for (flags of the batch) and never found:
// every positive score ends its reversed fill somewhere, so some launch left
// the pair out.
__host__ __device__ inline bool lost_begin(int score1, int read_begin1, uint32_t flags) {
    return (flags & (GSW_BEGIN | GSW_CIGAR)) && score1 > 0 && read_begin1 < 0;
}
// Counts a finished batch's records flagged kResInternal and flags those that
// lost their begins (small batches without CIGARs have no later stage that
// would see them).
cudaError_t launch_count_internal(const BatchView &b, unsigned long long *count, cudaStream_t st);

// Geometry of one class's launch: blocks resident on the SMs asked for, pairs
// in flight and scratch per block.
struct ClassGeom {
    int grid = 0, slots_per_block = 0;
    int cluster = 1;  // CTAs that share their pairs (the CTA classes)
    bool narrow = false;  // the CTA kernel of narrow strips
    size_t cm = 0, bnd = 0;  // bytes per slot
    size_t smem = 0;
    size_t bytes(int blocks) const {
        return (((size_t)blocks * slots_per_block * cm + 255) & ~(size_t)255) + (size_t)blocks * slots_per_block * bnd;
    }
};
// scratch bytes with which every class of fl.class_mask runs at full occupancy
size_t fill_scratch_want(const FillLaunch &fl, int sms);
// (a stream per kernel, as far as they go: kernels that share one wait for each
// other's longest pair)
constexpr int kSideStreams = 7;
struct SideStreams {
    cudaStream_t s[kSideStreams];
    cudaEvent_t fork, join[kSideStreams];
};
// Contexts whose kernels all go to the caller's stream, one after the other:
// those limited to some SMs, and those of a server.  A device has 8 hardware
// queues for its streams.  With 7 side streams a context, a server's streams
// share them, and a light batch's kernel waited in the queue behind a heavy
// batch's, several times a batch (10,000 requests/s of the mixed stream: short
// requests' p50 1,110 ms, in one stream 3.3 to 4.3; at 1,000/s p99 14 -> 1.0).
inline bool one_stream(int sms, int sms_all, bool shared) { return sms < sms_all || shared; }
// Side streams forked from `st`.  Whatever way their user leaves, `st` waits for
// what was queued on them: buffers are released in the order of `st`, so after
// a failed launch the kernels already queued beside it must not outlive them.
class SideFork {
public:
    SideFork(const SideStreams &aux, cudaStream_t st) : aux_(aux), st_(st) {}
    SideFork(const SideFork &) = delete;
    SideFork &operator=(const SideFork &) = delete;
    ~SideFork() { join(); }
    // the first n side streams wait for `st`
    cudaError_t fork(int n) {
        cudaError_t e = n > 0 ? cudaEventRecord(aux_.fork, st_) : cudaSuccess;
        for (; e == cudaSuccess && n_ < n; n_++)
            if ((e = cudaStreamWaitEvent(aux_.s[n_], aux_.fork, 0)) != cudaSuccess) break;
        return e;
    }
    // `st` waits for them (the host does where an event fails)
    cudaError_t join() {
        cudaError_t first = cudaSuccess;
        for (int k = 0; k < n_; k++) {
            cudaError_t e = cudaEventRecord(aux_.join[k], aux_.s[k]);
            if (e == cudaSuccess) e = cudaStreamWaitEvent(st_, aux_.join[k], 0);
            if (e != cudaSuccess) cudaStreamSynchronize(aux_.s[k]);
            if (first == cudaSuccess) first = e;
        }
        n_ = 0;
        return first;
    }

private:
    const SideStreams &aux_;
    cudaStream_t st_;
    int n_ = 0;
};
// one persistent launch per class in fl.class_mask, heaviest first, each with
// the slots its share of the scratch holds; side by side on `st` and the side
// streams (forked and joined by events) when the scratch holds all of them
cudaError_t launch_fill(const FillLaunch &fl, int sms, cudaStream_t st, const SideStreams &aux);
// Geometry and launch of one class, by kind of alphabet and lanes (one
// translation unit each, compiled in parallel: fill_dna.cu, fill_dna_half.cu,
// fill_general.cu, fill_general_half.cu)
#define GSW_FILL_UNITS(X) X(dna, true, false) X(dna_half, true, true) X(general, false, false) X(general_half, false, true)
#define GSW_DECLARE_UNIT(name, DNA, HALF)                                          \
    ClassGeom fill_geom_##name(int c, const FillLaunch &fl, int sms);              \
    cudaError_t fill_launch_##name(int c, const FillLaunch &fl, const ClassGeom &g, cudaStream_t st);
GSW_FILL_UNITS(GSW_DECLARE_UNIT)
#undef GSW_DECLARE_UNIT

// Geometry and launches of the allocation-free fill's two kernels (fill_static.cuh)
constexpr int kStaticMaxSmem = 200 << 10;
struct StaticGeom {
    size_t first_warp, first_smem;  // profile bytes of a warp and of a block of the first kernel
    int first_per_sm;               // its resident blocks per SM
    size_t rest_warp;               // profile bytes of a warp of the second kernel
    int rest_warps;                 // its warps per block
};
#define GSW_DECLARE_STATIC(name)                                                                            \
    StaticGeom static_geom_##name(int alphabet);                                                            \
    cudaError_t static_setup_##name();                                                                      \
    void static_launch_##name(bool rest, const BatchView &b, const Scoring &sc, uint8_t *scratch,           \
                              const StaticGeom &g, int grid, cudaStream_t st);
GSW_DECLARE_STATIC(dna)
GSW_DECLARE_STATIC(general)
#undef GSW_DECLARE_STATIC

struct PlanBuffers {
    int32_t *keys;       // [npairs]
    int32_t *hist;       // [kPlanBins]
    int32_t *cursor;     // [kPlanBins], after hist (cleared together)
    int32_t *binoff;     // [kPlanBins]
    int32_t *order;      // [npairs]
    int32_t *var_start;  // [kNumFillClasses+1]
    int32_t *task_lo;    // [kNumFillClasses]
    int32_t *task_hi;    // [kNumFillClasses]
    int32_t *ntasks;     // [1]
    int32_t *head;       // [kNumFillClasses]
};
int plan_launches(int npairs);  // kernels of one plan
// (a small batch's kPlanTrace plan also writes `need`, kNeedWords words)
cudaError_t launch_plan(const BatchView &b, const Scoring &sc, int32_t mode, const PlanBuffers &pb,
                        unsigned long long *need, cudaStream_t st);
bool plan_takes_needs(int npairs);

// Wide-band traceback (trace_ring.cu): banded global fill with direction
// bits on the CTA strip pipeline, then a warp walk per pair, group by group
// of pairs whose direction words fit the pool.
struct RingLaunchArgs {
    BatchView b;
    Scoring sc;
    const int32_t *order;     // plan order
    const int32_t *var_start; // class boundaries in `order`
    const long long *prefix;  // [n + 1] from launch_ring_needs
    int *final_h;             // [n]
    int *group;               // 3 ints: g0 (zeroed by the caller before the first group), g1, head
    uint32_t *pool;
    long long pool_words;
    int2 *bnd;                // boundary buffers: slots x bnd_stride int2
    long long bnd_stride;
    int slots;
    uint32_t *ops;            // walk: walk_warps x op_words
    long long op_words;
    int walk_warps;
    bool one_cta;             // no clusters (cluster_ctas)
};
int ring_trace_class();
int context_device(const gsw_ctx *ctx);
// Rounds a call's shapes (largest lengths, traceback scratch) up to powers of
// two, so that calls of similar shape repeat a captured pipeline (serving).
void context_set_graph_buckets(gsw_ctx *ctx, bool on);
// Other contexts' batches run beside this one's: its kernels keep to the
// caller's stream, and with one_cta to one CTA per pair (cluster_ctas).
void context_set_shared(gsw_ctx *ctx, bool on, bool one_cta);
int ring_slots_per_cta();
// prefix sums of the class's direction words; out[0] total, [1] max words of a pair, [2] max op words
cudaError_t launch_ring_needs(const BatchView &b, const Scoring &sc, const int32_t *order, const int32_t *var_start,
                              long long *prefix, unsigned long long *out, cudaStream_t st);
cudaError_t launch_ring_group(const RingLaunchArgs &a, int sms, cudaStream_t st);

struct TraceScratch {
    uint32_t *dirs;         // per warp: dir_words words (global direction bit-planes)
    int64_t dir_words;      // per warp
    uint32_t *ops;          // per warp: op_words words (reversed CIGAR runs)
    int64_t op_words;       // per warp
    const int32_t *order;   // pairs to trace: order[var_start[0] .. var_start[1])
    const int32_t *var_start;
};
int trace_block_threads();
// the needs (trace_needs) of a batch whose plan did not take them along, into
// zeroed words
cudaError_t launch_trace_need(const BatchView &b, const Scoring &sc, unsigned long long *need, cudaStream_t st);
// the classes in `mask`, one after the other
cudaError_t launch_trace_ad(const BatchView &b, const Scoring &sc, const TraceScratch &ts, int grid, unsigned mask,
                            cudaStream_t st);

// 16-bit full-rectangle traceback (trace16.cu), launch class v (t16_shape):
// direction and op words per group of P lanes, 32/P groups a warp
struct T16Scratch {
    uint32_t *dirs;
    int64_t dir_words;  // per group
    uint32_t *ops;
    int64_t op_words;   // per group
    const int32_t *order;
    const int32_t *var_start;
    int32_t *head;      // per-class task counters (zeroed by the plan)
    int warps;          // of the launch (the scratch holds 32/P groups each)
};
// warps of class v's launch that can be resident
int t16_max_warps(const Scoring &sc, int sms, int v);
cudaError_t launch_trace16(const BatchView &b, const Scoring &sc, const T16Scratch &ts, int sms, int v,
                           cudaStream_t st);

int band_block_threads();
// Grids and scratch of the three band classes (widths 8, 16, 32), each
// sized to the blocks that can be resident, scaled down to the budget.
struct BandGrids {
    int grid[3];
    int64_t words[3];  // per warp
    size_t off[3];     // byte offsets of the classes' scratch
    size_t total_bytes;
};
BandGrids band_grids(int rows_cap, int sms, size_t budget_bytes);
cudaError_t launch_band(const BatchView &b, const Scoring &sc, const PlanBuffers &pb, void *scratch,
                        const BandGrids &g, cudaStream_t st, const SideStreams &aux);

// small helpers (misc.cu)
// one pass over the pairs: [0, 1] largest lengths, [2, 3] arena extents,
// [4] nonzero if a length is outside [0, 2^24) or an offset negative,
// [5] 2^32 - 1 - the smallest query length (0 if any query or target is
// empty), [6] cells; the words are zero before
cudaError_t launch_batch_stats(const int64_t *q_off, const int32_t *q_len, const int64_t *t_off,
                               const int32_t *t_len, int32_t n, unsigned long long *out7, cudaStream_t st);
// 2-bit packed DNA letters to one byte per letter
cudaError_t launch_unpack2(const uint8_t *in, uint8_t *out, long long nletters, cudaStream_t st);
// (*bad is zero before)
cudaError_t launch_validate(const BatchView &b, const Scoring &sc, int32_t *bad, cudaStream_t st);
cudaError_t launch_fill_const(int32_t *dst, int32_t v, int32_t n, cudaStream_t st);
cudaError_t launch_fill_const64(int64_t *dst, int64_t v, int32_t n, cudaStream_t st);

}  // namespace gsw
