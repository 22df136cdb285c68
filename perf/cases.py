"""The work that users of the library have it do, as cases that can be timed.

Every case goes through the public entry points of the Python binding
(paper_1208_6350_gb300.gsw) or its Context, with seeded synthetic inputs of the
shapes the repository's workloads use.  ``prepare`` makes the inputs, ``run`` is
one call as a program makes it, ``work`` counts the bytes and the operations of
the method (ten two-input integer operations per cell of the forward matrix),
and ``exact`` computes the records by a plain column-by-column recurrence in
64-bit integers.
"""
import math

import numpy as np
import torch

from paper_1208_6350_gb300 import gsw
from paper_1208_6350_gb300 import workloads as wl

OPS_PER_CELL = 10
RECORD_BYTES = 48
BUDGET = 24 << 30  # device scratch of the program's one context

DNA = dict(match=2, mismatch=-2, gap_open=3, gap_extend=1)
DNA_LONG = dict(match=2, mismatch=-4, gap_open=4, gap_extend=2)
DNA_HIGH = dict(match=5, mismatch=-4, gap_open=10, gap_extend=1)
DNA_STRICT = dict(match=1, mismatch=-3, gap_open=2, gap_extend=2)


def listed():
    short = dict(kind="pairs", sub=0.01, indel=0.001, decoy=0.10, out="cigar", colmax=False, packed=False,
                 host=False, **DNA)
    return [
        # one read against one candidate window, as the README's example calls it
        dict(short, name="one_read_host", n=1, qmin=150, qmax=150, tmin=600, tmax=600, decoy=0.0, host=True),
        # a small batch of 100 nt reads with all outputs: latency of one batch
        dict(short, name="reads_1k", n=1000, qmin=100, qmax=100, tmin=1000, tmax=1000, sub=0.02, indel=0.002,
             decoy=0.0),
        # short-read extension at throughput, 2-bit packed arenas on the device, all outputs
        dict(short, name="extension_200k", n=200_000, qmin=100, qmax=250, tmin=300, tmax=1000, packed=True),
        # the same from host arrays (copies in and out included)
        dict(short, name="extension_host_20k", n=20_000, qmin=100, qmax=250, tmin=300, tmax=1000, host=True),
        # scores, ends and the per-column max arrays, no begins: filtering and scanning
        dict(short, name="score_colmax_30k", n=30_000, qmin=36, qmax=300, tmin=200, tmax=1500, out="score",
             colmax=True),
        # long reads at 10 % error, all outputs (tracebacks with wide bands)
        dict(kind="long", name="long_300", n=300, lmin=1000, lmax=20000, out="cigar", **DNA_LONG),
        # long reads whose scores leave 16 bits: the fills run again in 32-bit lanes
        dict(kind="long", name="long_high_scores_40", n=40, lmin=8000, lmax=16000, out="cigar", **DNA_HIGH),
        # protein queries against a database, all outputs
        dict(kind="protein", name="protein_40x1000", queries=40, db=1000, qmin=50, qmax=1000, out="cigar",
             gap_open=11, gap_extend=1),
        # one protein query kept as a profile against a database, scores and begins
        dict(kind="profile", name="profile_1x10000", qlen=350, db=10_000, out="begin", gap_open=11, gap_extend=1),
        # reads against a bacterial-size reference (windows, masks and end pairs)
        dict(kind="reference", name="reads_vs_5mb", n=200, qlen=100, ref=5_000_000, out="cigar", **DNA),
        # read overlaps: every pair of a set of 70 nt reads, scores and ends
        dict(kind="overlap", name="overlap_3000", n=3000, qlen=70, out="score", **DNA),
        # the allocation-free entry point
        dict(kind="static", name="static_8k", n=8192, qmin=100, qmax=250, tmin=300, tmax=1000, colmax=False, **DNA),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 0.49)))))))


def draw(rng):
    kind = rng.choice(["pairs", "pairs", "pairs", "long", "protein", "profile", "reference", "overlap", "static"])
    dna = dict(rng.choice([DNA, DNA, DNA_LONG, DNA_HIGH, DNA_STRICT]))
    if kind == "pairs":
        n = _log_int(rng, 1, 200_000)
        qmin = _log_int(rng, 30, 250)
        qmax = min(1000, max(qmin, _log_int(rng, qmin, 4 * qmin)))
        tmin = _log_int(rng, 100, 1000)
        tmax = max(tmin, _log_int(rng, tmin, 3 * tmin))
        most = 200_000 * 175 * 650  # cells of the largest listed batch
        n = max(1, min(n, int(most / (0.25 * (qmin + qmax) * (tmin + tmax)))))
        host = n <= 20_000 and rng.random() < 0.3
        out = rng.choice(["score", "begin", "cigar", "cigar"])
        return dict(kind=kind, n=n, qmin=qmin, qmax=qmax, tmin=tmin, tmax=tmax, sub=rng.choice([0.01, 0.02, 0.05]),
                    indel=rng.choice([0.001, 0.002, 0.01]), decoy=rng.choice([0.0, 0.1, 0.5]), out=out,
                    colmax=n <= 50_000 and rng.random() < 0.2, packed=rng.random() < 0.4, host=host, **dna)
    if kind == "long":
        lmin = _log_int(rng, 500, 6000)
        lmax = min(20000, _log_int(rng, lmin, 10 * lmin))
        n = max(2, min(_log_int(rng, 2, 300), int(300 * 8.0e7 / (1.2 * lmax * lmax))))
        return dict(kind=kind, n=n, lmin=lmin, lmax=lmax, out=rng.choice(["score", "cigar", "cigar"]),
                    **rng.choice([DNA_LONG, DNA, DNA_HIGH]))
    if kind == "protein":
        queries = _log_int(rng, 1, 40)
        qmin = _log_int(rng, 30, 300)
        return dict(kind=kind, queries=queries, db=_log_int(rng, 20, 1000), qmin=qmin,
                    qmax=min(1000, _log_int(rng, qmin, 1000)), out=rng.choice(["score", "begin", "cigar"]),
                    gap_open=rng.choice([10, 11, 12]), gap_extend=rng.choice([1, 2]))
    if kind == "profile":
        return dict(kind=kind, qlen=_log_int(rng, 40, 900), db=_log_int(rng, 100, 10_000),
                    out=rng.choice(["score", "begin"]), gap_open=11, gap_extend=rng.choice([1, 2]))
    if kind == "reference":
        return dict(kind=kind, n=_log_int(rng, 1, 200), qlen=_log_int(rng, 36, 100), ref=_log_int(rng, 5_000, 5_000_000),
                    out=rng.choice(["score", "begin", "cigar"]), **dna)
    if kind == "overlap":
        qlen = _log_int(rng, 36, 140)
        return dict(kind=kind, n=min(_log_int(rng, 50, 3000), int(3000 * 70 / qlen)), qlen=qlen,
                    out=rng.choice(["score", "score", "cigar"]) if qlen >= 60 else "score", **dna)
    tmin = _log_int(rng, 50, 500)
    return dict(kind="static", n=_log_int(rng, 1, 8192), qmin=30, qmax=_log_int(rng, 40, 400), tmin=tmin,
                tmax=_log_int(rng, tmin, 1000), colmax=rng.random() < 0.3, **dna)


# ------------------------------------------------------------------ inputs

_ctx = None
_stream = None


def _context():
    """The program's one context and the stream it calls on."""
    global _ctx, _stream
    if _ctx is None:
        _ctx = gsw.Context(0, BUDGET)
        _stream = torch.cuda.Stream()
    return _ctx, _stream


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _randint(g, lo, hi, n, dtype=torch.int64):
    return torch.randint(lo, hi, (n,), generator=g, device="cuda", dtype=dtype)


def _offsets(length):
    return torch.cumsum(length, 0) - length


def _ranges(start, length):
    """start[k], start[k] + 1, ... start[k] + length[k] - 1 for every k."""
    total = int(length.sum())
    base = torch.repeat_interleave(start - _offsets(length), length, output_size=total)
    return base + torch.arange(total, device="cuda")


def _mutated(g, src, length, sub, ins, dele, longest):
    """A copy of every sequence with substitutions, insertions of 1..longest
    random letters and deletions of 1..longest letters: (letters, lengths)."""
    n = src.numel()
    if n == 0:
        return src, length
    owner_seq = torch.repeat_interleave(torch.arange(len(length), device="cuda"), length, output_size=n)
    end = torch.cumsum(length, 0)[owner_seq]
    u = torch.rand(n, generator=g, device="cuda")
    k = _randint(g, 1, longest + 1, n)
    is_ins = (u >= sub) & (u < sub + ins)
    is_del = (u >= sub + ins) & (u < sub + ins + dele)
    other = ((src.long() + _randint(g, 1, 4, n)) % 4).to(torch.uint8)
    src = torch.where(u < sub, other, src)
    pos = torch.arange(n, device="cuda")
    diff = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    one = torch.ones(int(is_del.sum()), dtype=torch.int64, device="cuda")
    diff.index_add_(0, pos[is_del], one)
    diff.index_add_(0, torch.minimum(pos + k, end)[is_del], -one)
    kept = torch.cumsum(diff[:n], 0) == 0
    count = kept.long() + torch.where(is_ins, k, torch.zeros_like(k))
    total = int(count.sum())
    owner = torch.repeat_interleave(pos, count, output_size=total)
    rank = torch.arange(total, device="cuda") - _offsets(count)[owner]
    out = torch.where((rank == 0) & kept[owner], src[owner], _randint(g, 0, 4, total, torch.uint8))
    new_len = torch.zeros_like(length).index_add_(0, owner_seq, count)
    return out, new_len


def _dna_pairs(c, seed):
    """Queries, and targets that hold a mutated copy of the query at a random
    offset; a fraction of decoys are unrelated."""
    g = _gen(seed)
    n = c["n"]
    ql = _randint(g, c["qmin"], c["qmax"] + 1, n)
    tl = _randint(g, c["tmin"], c["tmax"] + 1, n)
    q = _randint(g, 0, 4, int(ql.sum()), torch.uint8)
    sub, indel = c.get("sub", 0.01), c.get("indel", 0.001)
    m, ml = _mutated(g, q, ql, sub, indel / 2, indel / 2, 3)
    true = torch.rand(n, generator=g, device="cuda") >= c.get("decoy", 0.1)
    keep = torch.minimum(ml, tl) * true
    t = _randint(g, 0, 4, int(tl.sum()), torch.uint8)
    room = ((tl - keep) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)).long()
    t[_ranges(_offsets(tl) + room, keep)] = m[_ranges(_offsets(ml), keep)]
    return q, ql, t, tl


def _long_pairs(c, seed):
    """Sources of log-uniform length; the query is the source at 10 % error,
    the target holds the source between random flanks, 1.2 times as long."""
    g = _gen(seed)
    n = c["n"]
    u = torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    sl = torch.exp(math.log(c["lmin"]) + u * math.log(c["lmax"] / c["lmin"])).round().long()
    s = _randint(g, 0, 4, int(sl.sum()), torch.uint8)
    q, ql = _mutated(g, s, sl, 0.06, 0.02, 0.02, 1)
    tl = (1.2 * sl.double()).round().long()
    t = _randint(g, 0, 4, int(tl.sum()), torch.uint8)
    room = ((tl - sl) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)).long()
    t[_ranges(_offsets(tl) + room, sl)] = s
    return q, ql, t, tl


def _database(g, n):
    """Lengths of a protein database: log-normal around 300, 20 to 5000."""
    z = torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    return torch.exp(math.log(300) + 0.6 * z).round().clamp(20, 5000).long()


def _protein_sets(g, ql, ndb):
    """Query and database arenas; every twentieth sequence of the database is
    a homolog of a query (40 % of its letters kept)."""
    q = _randint(g, 0, 20, int(ql.sum()), torch.uint8)
    dl = _database(g, ndb)
    hom = torch.arange(0, ndb, 20, device="cuda")
    of = _randint(g, 0, len(ql), len(hom))
    dl[hom] = ql[of]
    t = _randint(g, 0, 20, int(dl.sum()), torch.uint8)
    src = q[_ranges(_offsets(ql)[of], ql[of])]
    kept = torch.rand(len(src), generator=g, device="cuda") < 0.40
    at = _ranges(_offsets(dl)[hom], dl[hom])
    t[at] = torch.where(kept, src, t[at])
    return q, t, dl


def _matrix(c):
    if c["kind"] in ("protein", "profile"):
        return wl.synthetic_protein_matrix()
    return wl.dna_matrix(c["match"], c["mismatch"])


def _pack2(x):
    pad = torch.zeros((len(x) + 3) // 4 * 4, dtype=torch.uint8, device="cuda")
    pad[: len(x)] = x
    p = pad.view(-1, 4)
    return (p[:, 0] | (p[:, 1] << 2) | (p[:, 2] << 4) | (p[:, 3] << 6)).contiguous()


def _sequences(case, seed):
    """(query arena, its offsets and lengths, target arena, its offsets and
    lengths): one pair per row; for reads against a reference the targets are
    the reference, for overlaps both sides are the reads."""
    kind = case["kind"]
    if kind in ("pairs", "static"):
        q, ql, t, tl = _dna_pairs(case, seed)
        return q, _offsets(ql), ql, t, _offsets(tl), tl
    if kind == "long":
        q, ql, t, tl = _long_pairs(case, seed)
        return q, _offsets(ql), ql, t, _offsets(tl), tl
    g = _gen(seed)
    if kind == "protein":
        nq, nd = case["queries"], case["db"]
        ql = _randint(g, case["qmin"], case["qmax"] + 1, nq)
        q, t, dl = _protein_sets(g, ql, nd)
        a = torch.arange(nq, device="cuda").repeat_interleave(nd)
        b = torch.arange(nd, device="cuda").repeat(nq)
        return q, _offsets(ql)[a], ql[a], t, _offsets(dl)[b], dl[b]
    if kind == "profile":
        ql = torch.tensor([case["qlen"]], device="cuda")
        q, t, dl = _protein_sets(g, ql, case["db"])
        return q, torch.zeros_like(dl), ql.expand(len(dl)).contiguous(), t, _offsets(dl), dl
    n, m = case["n"], case["qlen"]
    ref = _randint(g, 0, 4, case["ref"] if kind == "reference" else max(m + 9, n * m // 10), torch.uint8)
    start = _randint(g, 0, len(ref) - m - 8, n)
    if kind == "reference":
        src = torch.full((n,), m + 8, dtype=torch.int64, device="cuda")
        q, ql = _mutated(g, ref[_ranges(start, src)], src, 0.01, 0.0005, 0.0005, 3)
        off = _offsets(ql)
        ql = ql.clamp(max=m)
        return q, off, ql, ref, torch.zeros_like(ql), torch.full_like(ql, len(ref))
    ln = torch.full((n,), m, dtype=torch.int64, device="cuda")
    q, _ = _mutated(g, ref[_ranges(start, ln)], ln, 0.01, 0.0, 0.0, 1)
    return q, _offsets(ln), ln, q, _offsets(ln), ln


def _flags(case):
    return {"score": 0, "begin": gsw.GSW_BEGIN, "cigar": gsw.GSW_CIGAR}[case.get("out", "score")]


def prepare(case, seed):
    kind = case["kind"]
    ctx, stream = _context()
    q, qo, ql, t, to, tl = _sequences(case, seed)
    s = dict(case=case, ctx=ctx, stream=stream, flags=_flags(case), W=_matrix(case), O=case["gap_open"],
             X=case["gap_extend"], n=len(ql))
    if kind == "pairs" and case["host"]:
        s.update(q=q.cpu().numpy(), t=t.cpu().numpy(), qo=qo.cpu().numpy(), to=to.cpu().numpy(),
                 ql=ql.int().cpu().numpy(), tl=tl.int().cpu().numpy(), cap=len(ql) * _words_per_pair(case) + 1024)
        s["words"] = np.zeros(s["cap"], np.uint32)
        s["cm"] = np.zeros(s["n"] * case["tmax"], np.int32)
        return s
    npairs = len(ql) * (len(ql) - 1) // 2 if kind == "overlap" else len(ql)
    s.update(q=q, t=t, qo=qo, to=to, ql=ql.int(), tl=tl.int(), npairs=npairs)
    if kind == "pairs" and case["packed"]:
        s.update(q=_pack2(q), t=_pack2(t), flags=s["flags"] | gsw.GSW_PACKED2)
    s["res"] = torch.zeros((npairs, RECORD_BYTES // 4), dtype=torch.int32, device="cuda")
    s["cap"] = 0
    if s["flags"] & gsw.GSW_CIGAR:
        s["cap"] = npairs * _words_per_pair(case) + 1024
        s["cigar"] = torch.zeros(s["cap"], dtype=torch.int32, device="cuda")
        s["words"] = torch.zeros(s["cap"], dtype=torch.int32, device="cuda")
        s["place"] = torch.arange(s["cap"], device="cuda")
    if case.get("colmax"):
        s["cmo"] = _offsets(tl)
        s["cm"] = torch.zeros(npairs * case["tmax"], dtype=torch.int32, device="cuda")
        s["flags"] |= gsw.GSW_COLMAX
    if kind == "profile":
        s["profile"] = _Profile(ctx, q.cpu().numpy(), s["W"], s["O"], s["X"])
    return s


def _words_per_pair(case):
    """CIGAR words reserved per pair: a gap in a few letters at most."""
    longest = case.get("lmax") or case.get("qmax") or case["qlen"]
    return 12 + longest // 4


class _Profile:
    def __init__(self, ctx, q, W, O, X):
        self.handle = gsw.gsw_profile_create(ctx.handle, q, W, O, X)

    def __del__(self):
        gsw.gsw_profile_destroy(self.handle)


# ------------------------------------------------------------------ the call

def _outputs(s):
    """Every field of the records but the place of the CIGAR words in the
    shared buffer, which no call fixes; the words follow in pair order."""
    res = s["res"]
    out = {"ends": res[:, :7], "cigar_len": res[:, 7], "flags": res[:, 10]}
    if "cm" in s:
        out["colmax"] = s["cm"]
    if s["flags"] & gsw.GSW_CIGAR:
        length = res[:, 7].clamp(min=0).long()
        if s["case"]["kind"] in ("overlap", "reference"):  # calls whose statistics cover their last batch only
            total = int(length.sum())
        else:
            total = gsw.gsw_last_stats(s["ctx"].handle)["cigar_words"]
        at = res.view(torch.int64)[:, 4] - torch.cumsum(length, 0) + length
        idx = torch.repeat_interleave(at, length, output_size=total) + s["place"][:total]
        torch.index_select(s["cigar"], 0, idx, out=s["words"][:total])
        out["cigar"] = s["words"]
    return out


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "pairs" and case["host"]:
        res, cig, (cm, _), _ = s["ctx"].align_host(s["q"], s["qo"], s["ql"], s["t"], s["to"], s["tl"], s["W"],
                                                   s["O"], s["X"], flags=s["flags"], colmax=case["colmax"],
                                                   cigar_capacity=s["cap"])
        out = {k: res[k] for k in ("score1", "score2", "ref_begin1", "ref_end1", "read_begin1", "read_end1",
                                   "ref_end2", "cigar_len", "flags")}
        if case["colmax"]:
            s["cm"][: len(cm)] = cm
            out["colmax"] = s["cm"]
        if s["flags"] & gsw.GSW_CIGAR:
            length = np.maximum(res["cigar_len"], 0).astype(np.int64)
            first = np.cumsum(length) - length
            idx = np.repeat(res["cigar_off"] - first, length) + np.arange(int(length.sum()))
            s["words"][: len(idx)] = cig[idx]
            out["cigar"] = s["words"]
        return out
    with torch.cuda.stream(s["stream"]):
        if kind == "static":
            rc = gsw.gsw_fill_static(s["n"], s["q"], s["qo"], s["ql"], s["t"], s["to"], s["tl"], case["tmax"], s["W"],
                                     s["O"], s["X"], flags=s["flags"], results=s["res"], colmax=s.get("cm"),
                                     colmax_off=s.get("cmo"), stream=s["stream"])
            if rc != gsw.GSW_OK:
                raise gsw.GswError(rc, "gsw_fill_static")
        elif kind == "profile":
            gsw.gsw_align_profile(s["ctx"].handle, s["profile"].handle, s["n"], s["t"], s["to"], s["tl"], s["flags"],
                                  results=s["res"], stream=s["stream"])
        elif kind == "reference":
            gsw.gsw_align_to_reference(s["ctx"].handle, s["n"], s["q"], s["qo"], s["ql"], s["t"], len(s["t"]), s["W"],
                                       s["O"], s["X"], flags=s["flags"], results=s["res"], cigar=s.get("cigar"),
                                       cigar_capacity=s["cap"], stream=s["stream"])
        elif kind == "overlap":
            rc = gsw.load().gsw_align_all_pairs(s["ctx"].handle, s["n"], s["q"].data_ptr(), s["qo"].data_ptr(),
                                                s["ql"].data_ptr(), s["W"].ctypes.data, 4, s["O"], s["X"], s["flags"],
                                                -1, 0, s["res"].data_ptr(),
                                                s["cigar"].data_ptr() if s["cap"] else None, s["cap"],
                                                s["stream"].cuda_stream)
            if rc != gsw.GSW_OK:
                raise gsw.GswError(rc, "gsw_align_all_pairs")
        else:
            gsw.gsw_align_batch(s["ctx"].handle, s["n"], s["q"], s["qo"], s["ql"], s["t"], s["to"], s["tl"], s["W"],
                                s["O"], s["X"], flags=s["flags"], results=s["res"], cigar=s.get("cigar"),
                                cigar_capacity=s["cap"], colmax=s.get("cm"), colmax_off=s.get("cmo"),
                                stream=s["stream"])
        return _outputs(s)


# ------------------------------------------------------------------ its work

def work(case):
    """Expected over the drawn lengths."""
    kind = case["kind"]
    mean_db = 300 * math.exp(0.18)
    if kind in ("pairs", "static"):
        n, m, t = case["n"], (case["qmin"] + case["qmax"]) / 2, (case["tmin"] + case["tmax"]) / 2
        cells, letters = n * m * t, n * (m + t)
    elif kind == "long":
        a, b = case["lmin"], max(case["lmax"], case["lmin"] + 1)
        n, r = case["n"], math.log(b / a)
        t = 1.2 * (b - a) / r
        cells, letters = n * 1.2 * (b * b - a * a) / (2 * r), n * 2.2 * (b - a) / r
    elif kind == "protein":
        m = (case["qmin"] + case["qmax"]) / 2
        n, t = case["queries"] * case["db"], mean_db
        cells, letters = n * m * mean_db, case["queries"] * m + case["db"] * mean_db
    elif kind == "profile":
        n, t = case["db"], mean_db
        cells, letters = n * case["qlen"] * mean_db, case["qlen"] + n * mean_db
    elif kind == "reference":
        n, t = case["n"], case["ref"]
        cells, letters = n * case["qlen"] * float(t), n * case["qlen"] + t
    else:
        n, t = case["n"] * (case["n"] - 1) // 2, case["qlen"]
        cells, letters = n * case["qlen"] * float(t), case["n"] * t
    if case.get("packed") and not case.get("host"):
        letters /= 4
    moved = letters + RECORD_BYTES * n + (24 * n if kind in ("pairs", "long", "static") else 0)
    if case.get("colmax"):
        moved += 4 * n * t + 8 * n
    return {"bytes": moved, "flops": OPS_PER_CELL * cells}


# ------------------------------------------------------------------ 64-bit values

def _columns(q, ql, t, tl, W, O, X, want_max):
    """Local affine-gap alignment of padded rows q [n, m] against t [n, k] in
    64-bit integers, column by column: (score, end column, end row, max array)."""
    n, m = q.shape
    far = -(1 << 40)
    dev = q.device
    row = torch.arange(m, device=dev)
    inside = row[None, :] < ql[:, None]
    H = torch.zeros((n, m), dtype=torch.int64, device=dev)
    E = torch.full((n, m), far, dtype=torch.int64, device=dev)
    best = torch.zeros(n, dtype=torch.int64, device=dev)
    end_t = torch.full_like(best, -1)
    end_q = torch.full_like(best, -1)
    cm = torch.zeros(t.shape, dtype=torch.int64, device=dev) if want_max else None
    table = torch.as_tensor(W, device=dev).long().reshape(-1)
    A = W.shape[0]
    for j in range(t.shape[1]):
        live = (j < tl)[:, None] & inside
        E = torch.maximum(E - X, H - O)
        D = torch.zeros_like(H)
        D[:, 1:] = H[:, :-1]
        T = torch.maximum(D + table[q * A + t[:, j: j + 1]], E).clamp(min=0)
        T = torch.where(live, T, torch.zeros_like(T))
        run_max = torch.cummax(T + X * row, 1).values
        F = torch.full_like(T, far)
        F[:, 1:] = run_max[:, :-1] - O - X * (row[1:] - 1)
        H = torch.where(live, torch.maximum(T, F), torch.zeros_like(T))
        top = H.max(1).values
        first = torch.where(H == top[:, None], row, m).min(1).values
        up = top > best
        best = torch.where(up, top, best)
        end_t = torch.where(up, torch.full_like(end_t, j), end_t)
        end_q = torch.where(up, first, end_q)
        if want_max:
            cm[:, j] = top
    return best, end_t, end_q, cm


def _padded(arena, off, length, step):
    """Rows arena[off + step * i], i < length, padded with letter 0."""
    m = max(1, int(length.max()))
    i = torch.arange(m, device="cuda")
    at = (off[:, None] + step * i[None, :]).clamp(0, max(0, len(arena) - 1))
    return torch.where(i[None, :] < length[:, None], arena[at].long(), 0)


def exact(case, seed):
    w = work(case)
    if case["kind"] in ("long", "reference", "overlap") or w["flops"] > 2e10:
        return None
    q, qo, ql, t, to, tl = _sequences(case, seed)
    W, O, X = _matrix(case), case["gap_open"], case["gap_extend"]
    parts, maxima = [], []
    size = max(1, int(2e7 / (max(1, int(ql.max())) + int(tl.max()))))
    for a in range(0, len(ql), size):
        k = slice(a, a + size)
        best, et, eq, cm = _columns(_padded(q, qo[k], ql[k], 1), ql[k], _padded(t, to[k], tl[k], 1), tl[k], W, O, X, True)
        col = torch.arange(cm.shape[1], device="cuda")
        half = torch.clamp(ql[k] // 2, min=15)
        masked = (best > 0)[:, None] & ((col[None, :] - et[:, None]).abs() <= half[:, None])
        rest = torch.where(masked, torch.zeros_like(cm), cm)
        second = rest.max(1).values
        at2 = torch.where(rest == second[:, None], col, cm.shape[1]).min(1).values
        at2 = torch.where(second > 0, at2, torch.full_like(at2, -1))
        bt, bq = torch.full_like(et, -1), torch.full_like(eq, -1)
        if _flags(case):
            _, rt, rq, _ = _columns(_padded(q, qo[k] + eq, eq + 1, -1), eq + 1, _padded(t, to[k] + et, et + 1, -1), et + 1,
                                    W, O, X, False)
            bt = torch.where(best > 0, et - rt, bt)
            bq = torch.where(best > 0, eq - rq, bq)
        parts.append(torch.stack([best, second, bt, et, bq, eq, at2], 1))
        if case.get("colmax"):
            maxima.append(cm[col[None, :] < tl[k][:, None]])
    ends = torch.cat(parts)
    maxima = torch.cat(maxima) if maxima else None
    if case.get("host"):
        names = ("score1", "score2", "ref_begin1", "ref_end1", "read_begin1", "read_end1", "ref_end2")
        out = {x: ends[:, i].contiguous() for i, x in enumerate(names)}
        out.update(cigar_len=None, flags=None)
    else:
        out = {"ends": ends, "cigar_len": None, "flags": None}
    if maxima is not None:
        whole = torch.zeros(case["n"] * case["tmax"], dtype=torch.int64, device="cuda")
        whole[: len(maxima)] = maxima
        out["colmax"] = whole
    if _flags(case) & gsw.GSW_CIGAR:
        out["cigar"] = None
    return out
