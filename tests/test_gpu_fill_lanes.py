"""The fill's lanes whose clamp is a half-precision multiply-add: taken when no
value of the batch's class can reach 2048 and O >= -(smallest matrix entry).
Every output against the oracle at the edges of that rule (all integers, so the
tolerance is zero)."""
import numpy as np
import pytest

from paper_1208_6350_gb300 import gsw
from paper_1208_6350_gb300 import workloads as wl
from parity_util import compare, run_gpu_host, run_oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    c = gsw.Context(0, 4 << 30)
    yield c
    c.close()


def batch(qs, ts, W, O, X, alphabet):
    ql, tl = np.array([len(x) for x in qs], np.int32), np.array([len(x) for x in ts], np.int32)
    off = lambda n: np.concatenate([[0], np.cumsum(n.astype(np.int64))[:-1]])
    return wl.Batch("lanes", np.concatenate(qs), off(ql), ql, np.concatenate(ts), off(tl), tl, W, O, X, alphabet)


def edge_batch(seed, rows, cols, W, O, X):
    """Exact copies (the largest scores), related and unrelated pairs, odd lengths."""
    rng = np.random.default_rng(seed)
    A = W.shape[0]
    top = int(np.argmax(np.diag(W)))
    qs, ts = [], []
    for k in range(24):
        m = rows if k < 4 else int(rng.integers(1, rows + 1))
        n = cols if k < 4 else int(rng.integers(1, cols + 1))
        q = np.full(m, top, np.uint8) if k % 4 == 0 else rng.integers(0, A, m).astype(np.uint8)
        t = rng.integers(0, A, n).astype(np.uint8)
        w = min(m, n)
        if k % 3 != 2:
            at = int(rng.integers(0, n - w + 1))
            t[at:at + w] = q[:w]
            if k % 3 == 1:
                t[rng.integers(0, n, max(1, n // 20))] = rng.integers(0, A)
        qs.append(q)
        ts.append(t)
    return batch(qs, ts, W, O, X, wl.DNA if A == 4 else wl.PROTEIN[:A])


# (match, mismatch, open, extend, rows): 7 * 291 + 7 + 3 = 2047 is the last row
# count whose values fit; O one below -mismatch keeps the biased lanes
@pytest.mark.parametrize("match,mismatch,O,X,rows", [
    (7, -3, 3, 1, 291), (7, -3, 3, 1, 292), (7, -3, 2, 1, 250), (1, -4, 4, 4, 256), (2, -2, 3, 0, 257),
    (127, -127, 127, 20, 14), (127, -127, 127, 20, 15), (1, 0, 0, 0, 120)])
def test_dna_lanes_at_the_edges_of_the_rule(ctx, match, mismatch, O, X, rows):
    for table in (None, [9] * 32, [13] * 32, [0] * 32):
        ctx.set_tune(table)
        try:
            b = edge_batch(match * 1000 + rows + O, rows, max(40, 2 * rows + 13), wl.dna_matrix(match, mismatch), O, X)
            compare(b, run_oracle(b), run_gpu_host(ctx, b))
        finally:
            ctx.set_tune(None)


@pytest.mark.parametrize("A,O,X,rows", [(20, 11, 1, 182), (20, 11, 1, 200), (5, 6, 2, 300), (20, 3, 1, 100)])
def test_general_alphabet_lanes(ctx, A, O, X, rows):
    W = np.ascontiguousarray(wl.synthetic_protein_matrix()[:A, :A])
    b = edge_batch(A + rows, rows, rows + 41, W, O, X)
    compare(b, run_oracle(b), run_gpu_host(ctx, b))


def _sized(n, rows, cols, seed, A=4):
    rng = np.random.default_rng(seed)
    qs = [rng.integers(0, A, int(rng.integers(max(1, rows - 31), rows + 1))).astype(np.uint8) for _ in range(n)]
    ts = []
    for q in qs:
        t = rng.integers(0, A, int(rng.integers(cols // 2, cols + 1))).astype(np.uint8)
        w = min(len(q), len(t))
        if rng.random() < 0.7:
            at = int(rng.integers(0, len(t) - w + 1))
            t[at:at + w] = q[:w]
        ts.append(t)
    W = wl.dna_matrix(2, -3) if A == 4 else np.ascontiguousarray(wl.synthetic_protein_matrix()[:A, :A])
    return batch(qs, ts, W, 5 if A == 4 else 11, 1, wl.DNA if A == 4 else wl.PROTEIN[:A])


# (pairs, longest query, longest target, alphabet): the 4-lane groups from
# 16,384 pairs, the 8-lane ones from 8,192, the tall 16-lane groups, several
# strips, and pairs heavy enough for the CTA class
@pytest.mark.parametrize("n,rows,cols,A", [
    (16384, 32, 40, 4), (16384, 48, 50, 4), (16400, 80, 90, 4), (16384, 112, 130, 4), (16384, 128, 60, 4),
    (8192, 129, 70, 4), (8191, 129, 70, 4), (300, 257, 300, 4), (300, 320, 200, 4), (300, 384, 401, 4),
    (200, 512, 300, 4), (200, 513, 300, 4), (8200, 100, 60, 20), (200, 321, 300, 20), (150, 512, 200, 20),
    (60, 900, 700, 20), (40, 1500, 900, 4)])
def test_classes_chosen_by_batch_size(ctx, n, rows, cols, A):
    b = _sized(n, rows, cols, n + rows, A)
    got = run_gpu_host(ctx, b)
    keep = np.random.default_rng(3).permutation(n)[:300]
    s = b.subset(keep)
    res, cig, (cm, off) = got
    compare(s, run_oracle(s), (res[keep], cig, (cm, off[keep])))


# the CTA class on clusters: more strips than warps, several pairs a cluster,
# 32-bit lanes, banded reversed strips, and a scratch that holds few CTAs
@pytest.mark.parametrize("n,lo,hi,match,O,X,budget_mb", [
    (1, 9000, 9000, 2, 4, 2, 4096), (7, 4000, 9000, 5, 10, 1, 4096), (60, 1800, 4200, 2, 4, 2, 4096),
    (5, 8000, 9000, 2, 4, 2, 256)])
def test_long_pairs_on_clusters(n, lo, hi, match, O, X, budget_mb):
    b = wl.dna_long_reads(n, lo, hi, match=match, mismatch=-4, gap_open=O, gap_extend=X, seed=n + lo)
    c = gsw.Context(0, budget_mb << 20)
    try:
        keep = np.arange(n)[:12]
        got = run_gpu_host(c, b, colmax=False)
    finally:
        c.close()
    s = b.subset(keep)
    compare(s, run_oracle(s, colmax=False), (got[0][keep], got[1], (None, None)), check_colmax=False)


# the 16-bit rectangle traceback's byte profiles: scores spanning at most 127
# (shifted bytes) and more (signed bytes), regions at the edges of its strips
@pytest.mark.parametrize("A,scale,O,X", [(20, 1, 11, 1), (20, 9, 40, 3), (3, 1, 4, 2), (32, 1, 9, 1)])
def test_general_alphabet_rectangle_traceback(ctx, A, scale, O, X):
    rng = np.random.default_rng(A * 100 + scale)
    W = rng.integers(-4, 2, (A, A))
    W = np.triu(W, 1) + np.triu(W, 1).T
    np.fill_diagonal(W, rng.integers(4, 9, A))
    W = np.ascontiguousarray((W * scale).astype(np.int8))
    qs, ts = [], []
    for m in (1, 63, 64, 65, 127, 128, 129, 255, 257, 300):
        q = rng.integers(0, A, m).astype(np.uint8)
        t = np.concatenate([q[: m // 2], rng.integers(0, A, 9 + m // 7), q[m // 2:]]).astype(np.uint8)
        mut = rng.random(len(t)) < 0.25
        t[mut] = rng.integers(0, A, int(mut.sum()))
        qs.append(q)
        ts.append(t)
    b = batch(qs, ts, W, O, X, "ABCDEFGHIJKLMNOPQRSTUVWXYZabcdef"[:A])
    compare(b, run_oracle(b), run_gpu_host(ctx, b))


# gsw_fill_static's two kernels: strips of 64 to 512 rows, taller queries, and
# scores beyond 16 bits, with max arrays
@pytest.mark.parametrize("A,match,O,X", [(4, 2, 3, 1), (4, 100, 30, 10), (20, 0, 11, 1)])
def test_static_fill_strip_heights(A, match, O, X):
    import torch
    W = wl.dna_matrix(match, -match) if A == 4 else wl.synthetic_protein_matrix()
    rng = np.random.default_rng(A + match)
    qs, ts = [], []
    for m in (1, 63, 64, 65, 128, 129, 192, 193, 256, 257, 320, 321, 384, 385, 512, 513, 700):
        q = rng.integers(0, A, m).astype(np.uint8)
        qs.append(q)
        ts.append(np.concatenate([rng.integers(0, A, 5), q, rng.integers(0, A, 9)]).astype(np.uint8))
    b = batch(qs, ts, W, O, X, wl.DNA if A == 4 else wl.PROTEIN)
    d = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (b.q, b.q_off, b.q_len, b.t, b.t_off, b.t_len)]
    cmo = np.concatenate([[0], np.cumsum(b.t_len.astype(np.int64))[:-1]])
    res = torch.zeros((b.npairs, 12), dtype=torch.int32, device="cuda")
    cm = torch.zeros(int(b.t_len.sum()), dtype=torch.int32, device="cuda")
    off = torch.from_numpy(cmo).cuda()
    torch.cuda.synchronize()
    rc = gsw.gsw_fill_static(b.npairs, *d, int(b.t_len.max()), W, O, X, flags=gsw.GSW_COLMAX, results=res, colmax=cm,
                             colmax_off=off)
    assert rc == gsw.GSW_OK
    r = res.cpu().numpy().view(gsw.RESULT_DTYPE).reshape(-1)
    compare(b, run_oracle(b), (r, None, (cm.cpu().numpy(), cmo)), check_begin=False, check_cigar=False)
