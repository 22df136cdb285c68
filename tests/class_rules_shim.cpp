// C entry points over the rules that choose a batch's kernels (gsw_impl.cuh),
// compiled by g++ for the CPU tests of those rules.
#include "gsw_impl.cuh"

namespace {
gsw::Scoring scoring(int A, const signed char *W, int O, int X) {
    gsw::Scoring sc{};
    sc.A = A;
    sc.O = O;
    sc.X = X;
    int mx = W[0], mn = W[0];
    for (int k = 0; k < A * A; ++k) {
        mx = W[k] > mx ? W[k] : mx;
        mn = W[k] < mn ? W[k] : mn;
        sc.W[k] = W[k];
    }
    sc.wmax = mx;
    sc.wmin = mn;
    sc.dna4 = A == 4;
    for (signed char &c : sc.fill_class) c = -1;
    return sc;
}
}  // namespace

extern "C" {

// (table: a tune table's classes, or null)
void cr_route_tuned(int A, const signed char *W, int O, int X, const signed char *table, int npairs, int minm, int maxm,
                    int maxn, double cells, int mode, int rows, int cols, unsigned *out) {
    gsw::Scoring sc = scoring(A, W, O, X);
    if (table)
        for (int b = 0; b < GSW_TUNE_BUCKETS; b++) sc.fill_class[b] = table[b];
    gsw::default_classes(sc, npairs, maxm, maxn, cells);
    out[0] = gsw::fill_class_mask(mode, maxm, sc, false, false, minm);
    const gsw::ClassRows r = gsw::fill_class_rows(mode, maxm, sc, out[0]);
    out[1] = gsw::fill_half_mask(r, maxn, sc);
    out[2] = gsw::fill_multi_mask(r);
    int v = mode == gsw::kFillForward ? gsw::pick_class16(rows, sc) : gsw::pick_class_reverse(rows, false, sc);
    if (gsw::cta_pair(v, rows, cols, sc, mode != gsw::kFillForward)) v = gsw::kClassLong16;
    out[3] = (unsigned)v;
    out[4] = (unsigned)gsw::variant_rows(v);
}

// What a batch of these sizes launches and where a pair of it goes: out[0] the
// launch mask, [1] the half-precision classes, [2] the classes with boundary
// rows, [3] the pair's class, [4] rows of that class's strip.
void cr_route(int A, const signed char *W, int O, int X, int npairs, int minm, int maxm, int maxn, double cells, int mode,
              int rows, int cols, unsigned *out) {
    cr_route_tuned(A, W, O, X, nullptr, npairs, minm, maxm, maxn, cells, mode, rows, cols, out);
}

int cr_half_fits(int A, const signed char *W, int O, int X, int rows, int cols) {
    return gsw::half_fits(rows, cols, scoring(A, W, O, X));
}

// trace class of a region, and whether a batch whose lengths reach maxm x maxn
// launches the wide-band kernel
int cr_trace(int A, const signed char *W, int O, int X, int maxm, int maxn, int la, int lb, int score1, int small,
             int *ring) {
    const gsw::Scoring sc = scoring(A, W, O, X);
    int dlo, dhi;
    *ring = gsw::ring_possible(maxm, maxn, sc);
    return gsw::trace_class(la, lb, score1, sc, small != 0, &dlo, &dhi);
}

// the 16-bit rectangle as a region of trace class `cls` launches it: scratch
// words, and the rows and columns it computes
void cr_rectangle(int A, int cls, int la, int lb, long long *out) {
    const int v = gsw::t16_launch_class(cls, la, A == 4) - gsw::kTraceT16First;
    const gsw::T16Shape s = gsw::t16_shape(v, A == 4);
    out[0] = s.need_words(la, lb);
    out[1] = (long long)s.strips(la) * s.rows();
    out[2] = lb + 2 * s.P;
}

int cr_cluster_alike(int npairs, int strips, int warps, int resident, int c) {
    return gsw::cluster_ctas_alike(npairs, strips, warps, resident, c);
}

int cr_one_stream(int sms, int sms_all, int shared) { return gsw::one_stream(sms, sms_all, shared != 0); }

int cr_cluster(int npairs, int few, int want, int most, int one_cta) {
    return gsw::cluster_ctas(npairs, few, want, most, one_cta != 0);
}

// class that a table of these values gives its bucket
int cr_tuned_class(int fill_class, float gcups, float gcups_default) {
    gsw_tune t = {};
    t.fill_class[7] = (signed char)fill_class;
    t.gcups[7] = gcups;
    t.gcups_default[7] = gcups_default;
    return gsw::tuned_class(t, 7);
}

int cr_consts(int which) {
    const int c[] = {gsw::kNumVariants, gsw::kVarP4First, gsw::kVarTallFirst, gsw::kTraceRingClass, gsw::kClassLong16};
    return c[which];
}

}  // extern "C"
