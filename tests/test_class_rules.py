"""The rules that choose a batch's kernels by its size, compiled from the
library's own header with g++ (tests/class_rules_shim.cpp): whatever class a
pair takes is one its batch launches, with the lanes and the boundary rows that
the pair needs, and a pair of the wide-band traceback is never left out.
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))
FORWARD, REVERSE = 0, 2


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if gxx is None or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("g++ or cuda_runtime.h not found")
    out = str(tmp_path_factory.mktemp("class_rules") / "libclassrules.so")
    subprocess.run([gxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-w", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1208_6350_gb300", "csrc"), "-I", inc,
                    os.path.join(HERE, "class_rules_shim.cpp"), "-o", out], check=True)
    L = ctypes.CDLL(out)
    P, i32 = ctypes.c_void_p, ctypes.c_int
    L.cr_route.argtypes = [i32, P, i32, i32, i32, i32, i32, i32, ctypes.c_double, i32, i32, i32, P]
    L.cr_route.restype = None
    L.cr_route_tuned.argtypes = [i32, P, i32, i32, P, i32, i32, i32, i32, ctypes.c_double, i32, i32, i32, P]
    L.cr_route_tuned.restype = None
    L.cr_half_fits.argtypes = [i32, P, i32, i32, i32, i32]
    L.cr_rectangle.argtypes = [i32, i32, i32, i32, P]
    L.cr_rectangle.restype = None
    L.cr_trace.argtypes = [i32, P, i32, i32, i32, i32, i32, i32, i32, i32, ctypes.POINTER(i32)]
    return L


def schemes():
    rng = np.random.default_rng(5)
    for match, mismatch, O, X in ((2, -3, 5, 2), (1, -1, 1, 1), (5, -4, 10, 1), (100, -100, 120, 10), (2, -6, 3, 1)):
        W = np.full((4, 4), mismatch, dtype=np.int8)
        np.fill_diagonal(W, match)
        yield W, O, X
    for A, O, X in ((20, 11, 1), (5, 4, 2), (24, 120, 3)):
        W = rng.integers(-4, 4, (A, A)).astype(np.int8)
        np.fill_diagonal(W, 9)
        yield W, O, X


def edge_lengths(rng, top):
    """Lengths at the edges of strips and buckets as well as in between."""
    edges = [x + d for x in (16, 48, 64, 96, 128, 256, 320, 384, 512, 1024, 1792, 4096) for d in (-1, 0, 1)]
    edges = [x for x in edges if x <= top] + [1, top]
    return int(rng.choice(edges)) if rng.random() < 0.5 else int(rng.integers(1, top + 1))


@pytest.mark.parametrize("mode", [FORWARD, REVERSE])
def test_every_pair_takes_a_launched_class_that_holds_it(lib, mode):
    rng = np.random.default_rng(17 + mode)
    nvar, p4, tall, _, long16 = (lib.cr_consts(k) for k in range(5))
    out = (ctypes.c_uint * 5)()
    seen = set()
    for W, O, X in schemes():
        p, A = W.ctypes.data_as(ctypes.c_void_p), len(W)
        for _ in range(400):
            npairs = int(rng.choice([1, 40, 2047, 2048, 8191, 8192, 16383, 16384, 300000]))
            maxm, maxn = edge_lengths(rng, 6000), edge_lengths(rng, 40000)
            minm = int(rng.integers(1, maxm + 1))
            rows = int(rng.choice([minm, maxm, rng.integers(minm, maxm + 1)])) if mode == FORWARD \
                else edge_lengths(rng, maxm)
            cols = int(rng.choice([1, maxn, rng.integers(1, maxn + 1)]))
            cells = float(npairs) * rng.random() * maxm * maxn
            lib.cr_route(A, p, O, X, npairs, minm, maxm, maxn, cells, mode, rows, cols, out)
            mask, half, multi, v, strip = out
            what = (A, npairs, minm, maxm, maxn, rows, cols, v)
            assert (mask >> v) & 1, what
            if (half >> v) & 1:
                assert lib.cr_half_fits(A, p, O, X, rows, cols), what
            if rows > strip:
                assert (multi >> v) & 1, what
            if p4 <= v < tall:  # four lanes: DNA, one strip, half-precision lanes only
                assert A == 4 and rows <= strip and (half >> v) & 1 and npairs >= 16384, what
            seen.add(v)
    # (the classes the default rule can choose: 4 and 8 lanes go forward only)
    assert long16 in seen and any(tall <= v < nvar for v in seen)
    assert any(p4 <= v < tall for v in seen) == (mode == FORWARD)


def test_a_tune_table_keeps_the_classes_it_names(lib):
    # classes 0..6 and 9..13 run a longer query strip after strip, whatever the
    # batch's size; a 4-letter query of several strips reverses on a CTA
    rng = np.random.default_rng(29)
    p8, long16, buckets = 8, lib.cr_consts(4), 32
    out = (ctypes.c_uint * 5)()
    several = 0
    for W, O, X in schemes():
        p, A = W.ctypes.data_as(ctypes.c_void_p), len(W)
        for _ in range(300):
            table = rng.choice([-1, 0, 1, 2, 3, 4, 5, 6, 8, 9, 10, 11, 12, 13], buckets).astype(np.int8)
            t = table.ctypes.data_as(ctypes.c_void_p)
            npairs = int(rng.choice([1, 160, 8192, 300000]))
            maxm, maxn = edge_lengths(rng, 1024), edge_lengths(rng, 40000)
            rows, cols = edge_lengths(rng, maxm), int(rng.choice([1, maxn]))
            code = int(table[(rows - 1) // 32])
            if code < 0:
                continue
            named = long16 if code == 8 else (p8 + code - 9 if code >= 9 else code)
            for mode in (FORWARD, REVERSE):
                lib.cr_route_tuned(A, p, O, X, t, npairs, 1, maxm, maxn, float(npairs) * maxm * maxn, mode, rows, cols, out)
                mask, half, multi, v, strip = out
                what = (A, npairs, maxm, maxn, rows, cols, code, mode, v)
                assert (mask >> v) & 1, what
                if v != named:
                    assert mode == REVERSE and A == 4 and v == long16, what
                elif rows > strip:
                    several += named != long16
                    assert (multi >> v) & 1, what
    assert several > 100


def test_large_batches_run_several_strips_in_groups(lib):
    # 20,000 pairs of 540 to 1,400 x 600 to 1,000 (compared with the oracle in
    # tests/test_gpu_large_batches.py): no query goes to a CTA, and the classes
    # of 320 to 512 rows are among those of several strips
    tall, nvar = lib.cr_consts(2), lib.cr_consts(0)
    out = (ctypes.c_uint * 5)()
    seen = {}
    for A, match, mismatch, O, X in ((4, 1, -3, 5, 2), (4, 5, -4, 10, 1), (20, 6, -2, 11, 1)):
        W = np.full((A, A), mismatch, np.int8)
        np.fill_diagonal(W, match)
        for rows in range(540, 1401):
            lib.cr_route(A, W.ctypes.data_as(ctypes.c_void_p), O, X, 20_000, 540, 1400, 1000, 20_000 * 970.0 * 800.0,
                         FORWARD, rows, 1000, out)
            _, half, _, v, strip = out
            assert v < nvar and rows > strip, (A, rows, v)
            seen.setdefault((A, match, bool((half >> v) & 1)), set()).add(v)
    assert (4, 1, True) in seen and (4, 5, False) in seen and (20, 6, False) in seen
    assert all(any(v >= tall for v in s) and any(v < tall for v in s) for s in seen.values()), seen


def test_even_batches_of_many_pairs_stay_in_groups(lib):
    long16 = lib.cr_consts(4)
    out = (ctypes.c_uint * 5)()

    def route(A, npairs, rows, cols, share):
        # a pair of the batch's largest lengths; share: mean cells over its cells
        W = np.full((A, A), -2, np.int8)
        np.fill_diagonal(W, 3)
        lib.cr_route(A, W.ctypes.data_as(ctypes.c_void_p), 5, 2, npairs, 1, rows, cols, share * npairs * rows * cols,
                     FORWARD, rows, cols, out)
        assert (out[0] >> out[3]) & 1
        return out[3]

    for rows, cols in ((1000, 1000), (1500, 1200)):
        assert route(4, 4000, rows, cols, 0.5) == long16   # the chip part empty
        assert route(4, 4864, rows, cols, 0.5) == long16
        assert route(4, 4865, rows, cols, 0.5) != long16   # a group for every pair, and more pairs
        assert route(4, 4865, rows, cols, 0.05) == long16  # a few pairs far above the others
    assert route(20, 2432, 900, 800, 0.5) == long16
    assert route(20, 2433, 900, 800, 0.5) != long16
    assert route(20, 2433, 1025, 800, 0.5) == long16
    assert route(20, 9000, 1025, 800, 0.5) == long16
    assert route(20, 8192, 1000, 800, 0.5) != long16 and route(20, 8193, 1000, 800, 0.5) == long16
    assert route(20, 8193, 700, 800, 0.5) != long16


def test_wide_bands_are_never_left_out(lib):
    rng = np.random.default_rng(23)
    ring_class = lib.cr_consts(3)
    ring = ctypes.c_int()
    wide = without = 0
    for W, O, X in schemes():
        p, A = W.ctypes.data_as(ctypes.c_void_p), len(W)
        for _ in range(6000):
            top = int(rng.choice([300, 600, 2000, 9000, 40000]))
            maxm, maxn = edge_lengths(rng, top), edge_lengths(rng, top)
            la = int(rng.choice([1, maxm, edge_lengths(rng, maxm)]))
            lb = int(rng.choice([1, maxn, edge_lengths(rng, maxn)]))
            score = int(rng.integers(1, max(2, min(la, lb) * int(W.max()) + 1)))
            cls = lib.cr_trace(A, p, O, X, maxm, maxn, la, lb, score, int(rng.integers(0, 2)), ctypes.byref(ring))
            assert cls != ring_class or ring.value, (A, O, X, maxm, maxn, la, lb, score)
            wide += cls == ring_class
            without += not ring.value
    assert wide and without


def test_rectangles_fit_the_shape_that_runs_them(lib):
    # scratch of a class within its allowance, and every value of the padded
    # rectangle within a biased 16-bit lane, in the strips and groups launched
    rng = np.random.default_rng(31)
    out = (ctypes.c_longlong * 3)()
    ring = ctypes.c_int()
    tall = large = 0
    for W, O, X in list(schemes()) + [(np.full((20, 20), 2, np.int8), 11, 10), (np.full((24, 24), 40, np.int8), 5, 2)]:
        p, A = W.ctypes.data_as(ctypes.c_void_p), len(W)
        for _ in range(4000):
            la, lb = edge_lengths(rng, 4096), edge_lengths(rng, 4096)
            score = int(rng.integers(1, max(2, min(la, lb) * max(int(W.max()), 1) + 1)))
            cls = lib.cr_trace(A, p, O, X, la, lb, la, lb, score, int(rng.integers(0, 2)), ctypes.byref(ring))
            if cls < 5:
                continue
            lib.cr_rectangle(A, cls, la, lb, out)
            words, rows, cols = out
            what = (A, O, X, la, lb, cls, words, rows, cols)
            assert words <= (1 << 17 if A == 4 or cls == 5 else 1 << 20), what
            assert 3 * O + X * (rows + cols + 2) - min(0, int(W.min())) <= 30000, what
            assert int(W.max()) * (min(rows, cols) + 1) <= 30000, what
            tall += A != 4 and la > 256
            large += cls == 6 and A != 4
    assert tall and large


def test_side_streams_only_where_a_context_has_the_device_to_itself(lib):
    assert not lib.cr_one_stream(152, 152, 0)
    assert lib.cr_one_stream(133, 152, 0)  # limited to some SMs
    assert lib.cr_one_stream(152, 152, 1) and lib.cr_one_stream(133, 152, 1)  # a server's


def test_clusters_only_where_a_batch_has_the_chip_to_itself(lib):
    for npairs in (1, 40, 2048, 2049, 10_000):
        for want in (0, 1, 2, 3, 5, 8, 40):
            c = lib.cr_cluster(npairs, 2048, want, 8, 0)
            if npairs > 2048 or want <= 1:
                assert c == 1
            else:
                assert c == min(8, 1 << (want - 1).bit_length()), (npairs, want, c)
            assert lib.cr_cluster(npairs, 2048, want, 8, 1) == 1  # a server's heavy worker
    assert lib.cr_cluster(300, 2048, 4, 4, 0) == 4


def test_a_saved_tune_table_installs_what_was_tuned(lib, monkeypatch):
    from paper_1208_6350_gb300 import gsw
    lib.cr_tuned_class.argtypes = [ctypes.c_int, ctypes.c_float, ctypes.c_float]
    rng = np.random.default_rng(37)
    named = rng.choice([0, 1, 2, 3, 4, 5, 6, 8, 9, 10, 11, 12, 13], gsw.TUNE_BUCKETS).astype(int)
    rule = rng.uniform(1000, 4000, gsw.TUNE_BUCKETS).astype(np.float32)
    own = np.where(np.arange(gsw.TUNE_BUCKETS) % 3 == 0, rule, rule + np.float32(0.01))  # the rule wins every third
    want = [-1 if b % 3 == 0 else int(named[b]) for b in range(gsw.TUNE_BUCKETS)]
    assert [lib.cr_tuned_class(int(named[b]), own[b], rule[b]) for b in range(gsw.TUNE_BUCKETS)] == want
    # a table without rates (made by hand), or one that names the default rule
    assert lib.cr_tuned_class(9, 0.0, 0.0) == 9 and lib.cr_tuned_class(-1, 0.0, 0.0) == -1

    class Lib:  # stands in for the library: a tuned table, and what is installed
        def gsw_autotune(self, ctx, m, a, o, x, n, out):
            t = out._obj
            for b in range(gsw.TUNE_BUCKETS):
                t.fill_class[b], t.gcups[b], t.gcups_default[b] = int(named[b]), own[b], rule[b]
            return gsw.GSW_OK

        def gsw_context_set_tune(self, ctx, table):
            t = table._obj
            self.table = [lib.cr_tuned_class(t.fill_class[b], t.gcups[b], t.gcups_default[b])
                          for b in range(gsw.TUNE_BUCKETS)]
            return gsw.GSW_OK

    fake = Lib()
    monkeypatch.setattr(gsw, "load", lambda: fake)
    ctx = gsw.Context.__new__(gsw.Context)
    ctx.handle = None
    t = ctx.autotune(np.eye(4, dtype=np.int8), 1, 1)
    for saved in (t, t["installed"]):
        ctx.set_tune(saved)
        assert fake.table == want
    assert t["fill_class"] == named.tolist()
    ctx.set_tune(t["fill_class"])  # the classes alone: as named
    assert fake.table == named.tolist()


def test_clusters_of_like_pairs_run_the_fewest_rounds(lib):
    alike = lib.cr_cluster_alike
    # 456 CTAs of 4 warps; 5 strips: two rounds either way, then three against two
    assert alike(300, 5, 4, 456, 2) == 1 and alike(500, 5, 4, 456, 2) == 2 and alike(800, 5, 4, 456, 2) == 1
    assert alike(40, 20, 4, 456, 8) == 8 and alike(1, 20, 4, 456, 8) == 8 and alike(1, 4, 4, 456, 1) == 1
    rng = np.random.default_rng(41)
    for _ in range(2000):
        n, s, r, c = (int(rng.integers(1, x)) for x in (2100, 40, 500, 9))
        x = alike(n, s, 4, r, c)
        assert 1 <= x <= c and x & (x - 1) == 0
        rounds = lambda y: -(-(-(-n // max(r // y, 1)) * s) // (4 * y))
        assert all(rounds(x) < rounds(y) or (rounds(x) == rounds(y) and x <= y) for y in (1, 2, 4, 8) if y <= c)
