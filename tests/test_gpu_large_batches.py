"""Kernel forms that only large batches take, against the oracle (all integers,
so the tolerance is zero): the wide-band traceback's 16-row strips and the CTA
fill without clusters (more than 2,048 pairs), several pairs opened in a phase,
and group fills of several strips (batches in which no pair's strips take a
large part of the time)."""
import numpy as np
import pytest

from paper_1208_6350_gb300 import gsw
from paper_1208_6350_gb300 import workloads as wl
from parity_util import compare, run_gpu_device, run_oracle

pytestmark = pytest.mark.gpu


def make(qs, ts, W, O, X):
    ql, tl = np.array([len(x) for x in qs], np.int32), np.array([len(x) for x in ts], np.int32)
    off = lambda n: np.concatenate([[0], np.cumsum(n.astype(np.int64))[:-1]])
    return wl.Batch("large", np.concatenate(qs), off(ql), ql, np.concatenate(ts), off(tl), tl, W, O, X,
                    wl.DNA if len(W) == 4 else wl.PROTEIN)


def part(b, idx):
    """The batch of the pairs `idx` alone."""
    cut = lambda a, o, n: [a[int(o[p]):int(o[p]) + int(n[p])] for p in idx]
    return make(cut(b.q, b.q_off, b.q_len), cut(b.t, b.t_off, b.t_len), b.W, b.gap_open, b.gap_extend)


def check(b, got, idx):
    """Compares the pairs `idx` of a whole batch's outputs."""
    res, cig, (cm, off) = got
    s = part(b, idx)
    words = [cig[int(res["cigar_off"][p]):int(res["cigar_off"][p]) + max(int(res["cigar_len"][p]), 0)] for p in idx]
    r = res[idx].copy()
    r["cigar_off"] = np.concatenate([[0], np.cumsum([len(w) for w in words])[:-1]])
    compare(s, run_oracle(s), (r, np.concatenate(words) if words else cig[:0],
                               (np.concatenate([cm[off[p]:off[p] + int(b.t_len[p])] for p in idx]), s.t_off)))


def short_pairs(rng, n):
    for _ in range(n):
        t = rng.integers(0, 4, int(rng.integers(40, 90))).astype(np.uint8)
        q = t[3:3 + int(rng.integers(20, 36))].copy()
        q[rng.integers(0, len(q))] = rng.integers(0, 4)
        yield q, t


def long_pairs(rng, n, lo, hi, gap):
    """Related pairs whose alignments hold gaps of up to `gap` letters: bands of
    more than 512 diagonals."""
    for _ in range(n):
        s = rng.integers(0, 4, int(rng.integers(lo, hi + 1))).astype(np.uint8)
        cut, g = int(rng.integers(len(s) // 3, len(s) // 2)), int(rng.integers(gap // 2, gap + 1))
        q = np.concatenate([s[:cut], rng.integers(0, 4, g).astype(np.uint8), s[cut:]])
        cut = int(rng.integers(len(s) // 2, 2 * len(s) // 3))
        t = np.concatenate([s[:cut], rng.integers(0, 4, g).astype(np.uint8), s[cut:]])
        q[rng.integers(0, len(q), len(q) // 25)] = rng.integers(0, 4)
        yield q, t


@pytest.fixture(scope="module")
def wide():
    rng = np.random.default_rng(71)
    pairs = list(short_pairs(rng, 2049)) + list(long_pairs(rng, 36, 1500, 3200, 350))
    order = rng.permutation(len(pairs))
    b = make([pairs[p][0] for p in order], [pairs[p][1] for p in order], wl.dna_matrix(2, -4), 4, 2)
    return b, run_oracle(b)


def test_wide_bands_of_a_large_batch_in_one_pool_group(wide):
    b, ora = wide
    c = gsw.Context(0, 4 << 30)
    try:
        compare(b, ora, run_gpu_device(c, b))
        st = gsw.gsw_last_stats(c.handle)
        assert st["ring_groups"] == 1 and st["ring_words"] > 36 << 17
        whole = 4 * st["ring_words"]
    finally:
        c.close()
    # a budget whose share for the direction words holds a part of them
    c = gsw.Context(0, (180 << 20) + whole)
    try:
        compare(b, ora, run_gpu_device(c, b))
        assert gsw.gsw_last_stats(c.handle)["ring_groups"] >= 2
    finally:
        c.close()


def test_cta_fill_without_clusters():
    # 8 SMs hold 24 CTAs of the DNA fill: 300 pairs of several strips are more
    # than 4 per CTA, and with them 2,049 short ones, so no clusters
    rng = np.random.default_rng(73)
    pairs = list(short_pairs(rng, 2049))
    for _ in range(300):
        t = rng.integers(0, 4, int(rng.integers(200, 700))).astype(np.uint8)
        q = rng.integers(0, 4, int(rng.integers(1793, 2400))).astype(np.uint8)
        at = int(rng.integers(0, len(q) - len(t)))
        q[at:at + len(t)] = t
        q[rng.integers(0, len(q), len(q) // 20)] = rng.integers(0, 4)
        pairs.append((q, t))
    b = make([p[0] for p in pairs], [p[1] for p in pairs], wl.dna_matrix(2, -3), 5, 2)
    c = gsw.Context(0, 4 << 30)
    try:
        assert gsw.load().gsw_context_set_sm_limit(c.handle, 8) == gsw.GSW_OK
        compare(b, run_oracle(b), run_gpu_device(c, b))
    finally:
        c.close()


def test_cta_fill_opens_its_share_of_like_pairs():
    # 2,100 pairs of two strips, nearly alike, on the 24 CTAs of 8 SMs: as many
    # at once as a CTA has slots
    rng = np.random.default_rng(77)
    pairs = []
    for _ in range(2100):
        t = rng.integers(0, 4, int(rng.integers(290, 321))).astype(np.uint8)
        q = rng.integers(0, 4, int(rng.integers(1800, 1851))).astype(np.uint8)
        at = int(rng.integers(0, len(q) - len(t)))
        q[at:at + len(t)] = t
        q[rng.integers(0, len(q), len(q) // 20)] = rng.integers(0, 4)
        pairs.append((q, t))
    b = make([p[0] for p in pairs], [p[1] for p in pairs], wl.dna_matrix(2, -3), 5, 2)
    c = gsw.Context(0, 4 << 30)
    try:
        assert gsw.load().gsw_context_set_sm_limit(c.handle, 8) == gsw.GSW_OK
        check(b, run_gpu_device(c, b), np.sort(rng.choice(2100, 300, replace=False)))
    finally:
        c.close()


@pytest.mark.parametrize("n", [2048, 2049, 4096, 4097, 16383, 16384])
def test_plans_by_one_block_or_the_chip(n):
    rng = np.random.default_rng(83 + n)
    pairs = list(short_pairs(rng, n))
    pairs[0] = (pairs[0][0][:0], pairs[0][1])  # an empty query and an empty target
    pairs[n - 1] = (pairs[n - 1][0], pairs[n - 1][1][:0])
    b = make([p[0] for p in pairs], [p[1] for p in pairs], wl.dna_matrix(2, -3), 5, 2)
    c = gsw.Context(0, 2 << 30)
    try:
        check(b, run_gpu_device(c, b), np.unique(np.concatenate([[0, n - 1], rng.choice(n, 600)])))
    finally:
        c.close()


@pytest.mark.parametrize("A,match,mismatch,O,X", [(4, 1, -3, 5, 2), (4, 5, -4, 10, 1), (20, 0, 0, 11, 1)])
def test_group_fills_of_several_strips(A, match, mismatch, O, X):
    # 20,000 pairs of 540 to 1,400 rows (tests/test_class_rules.py: what such a
    # batch launches), values inside and outside the half-precision lanes
    rng = np.random.default_rng(79 + A + match)
    W = wl.dna_matrix(match, mismatch) if A == 4 else wl.synthetic_protein_matrix()
    n = 20_000
    ql, tl = rng.integers(540, 1401, n).astype(np.int32), rng.integers(600, 1001, n).astype(np.int32)
    off = lambda x: np.concatenate([[0], np.cumsum(x.astype(np.int64))[:-1]])
    q, t = (rng.integers(0, A, int(x.sum())).astype(np.uint8) for x in (ql, tl))
    qo, to = off(ql), off(tl)
    idx = np.sort(rng.choice(n, 240, replace=False))
    for k, p in enumerate(idx):  # related pairs among those compared, exact copies too
        w = int(min(ql[p], tl[p]))
        at = int(rng.integers(0, ql[p] - w + 1))
        if k % 4 == 3:
            continue
        piece = t[to[p]:to[p] + w].copy()
        if k % 4:
            piece[rng.integers(0, w, max(1, w // 12))] = rng.integers(0, A)
        q[qo[p] + at:qo[p] + at + w] = piece
    b = wl.Batch("strips", q, qo, ql, t, to, tl, W, O, X, wl.DNA if A == 4 else wl.PROTEIN)
    c = gsw.Context(0, 8 << 30)
    try:
        check(b, run_gpu_device(c, b), idx)
    finally:
        c.close()
