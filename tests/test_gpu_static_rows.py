"""gsw_fill_static's queries of more than 512 rows against the oracle (all
integers, so the tolerance is zero): whole warps over one strip of 640 or 1,024
rows, several strips and 32-bit lanes in the second kernel, beside shorter and
empty ones in the first."""
import numpy as np
import pytest

from paper_1208_6350_gb300 import gsw
from paper_1208_6350_gb300 import workloads as wl
from parity_util import compare, run_oracle

pytestmark = pytest.mark.gpu

TALL = (512, 513, 640, 641, 1023, 1024, 1025, 1100, 2048, 2049, 3000)


@pytest.mark.parametrize("A,match,O,X", [(4, 1, 3, 1), (4, 2, 3, 1), (4, 100, 30, 10), (20, 0, 11, 1)])
@pytest.mark.parametrize("mix", ["tall", "mixed"])
def test_static_fill_of_tall_queries(A, match, O, X, mix):
    import torch
    W = wl.dna_matrix(match, -match) if A == 4 else wl.synthetic_protein_matrix()
    rng = np.random.default_rng(10 * A + match)
    rows = list(TALL) * 2
    if mix == "mixed":
        rows += [0, 1, 64, 65, 130, 250, 257, 300, 333, 400] * 3 + [700] * 9
    rng.shuffle(rows)
    qs, ts = [], []
    for k, m in enumerate(rows):
        n = int(rng.choice([1, 3, 31, 700, 1021, 1024])) if k % 3 else int(rng.integers(600, 1025))
        q, t = rng.integers(0, A, m).astype(np.uint8), rng.integers(0, A, n).astype(np.uint8)
        w = min(m, n)
        if k % 4 and w:  # related pairs, every other one with substitutions
            piece = q[m - w:].copy()
            if k % 2:
                piece[rng.integers(0, w, max(1, w // 15))] = rng.integers(0, A)
            t[n - w:] = piece
        qs.append(q)
        ts.append(t)
    ts[len(ts) // 2] = ts[len(ts) // 2][:0]
    ql, tl = np.array([len(x) for x in qs], np.int32), np.array([len(x) for x in ts], np.int32)
    off = lambda x: np.concatenate([[0], np.cumsum(x.astype(np.int64))[:-1]])
    b = wl.Batch("static", np.concatenate(qs), off(ql), ql, np.concatenate(ts), off(tl), tl, W, O, X,
                 wl.DNA if A == 4 else wl.PROTEIN)
    d = [torch.from_numpy(np.ascontiguousarray(x)).cuda() for x in (b.q, b.q_off, b.q_len, b.t, b.t_off, b.t_len)]
    res = torch.full((b.npairs, 12), -7, dtype=torch.int32, device="cuda")
    cm = torch.full((int(tl.sum()),), -7, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    rc = gsw.gsw_fill_static(b.npairs, *d, int(tl.max()), W, O, X, flags=gsw.GSW_COLMAX, results=res, colmax=cm,
                             colmax_off=torch.from_numpy(b.t_off).cuda())
    assert rc == gsw.GSW_OK
    r = res.cpu().numpy().view(gsw.RESULT_DTYPE).reshape(-1)
    compare(b, run_oracle(b), (r, None, (cm.cpu().numpy(), b.t_off)), check_begin=False, check_cigar=False)
