"""Warp-per-hit traceback at the edges of its lanes, row counts (4 and 8 rows
per lane), bands and 8-step decision words, against the oracle's walk."""
import numpy as np
import pytest

import oracle
from paper_1701_01575_gb300 import dsa
from paper_1701_01575_gb300 import workloads as W

from test_gpu_parity import check_traceback

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1701_01575_gb300 import build
    build.build()
    c = dsa.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("mode,fe", [(dsa.LOCAL, 15), (dsa.GLOBAL, 15), (dsa.SEMIGLOBAL, 15),
                                     (dsa.SEMIGLOBAL, 12), (dsa.SEMIGLOBAL, 3), (dsa.SEMIGLOBAL, 5)])
def test_lane_band_and_word_edges(ctx, mode, fe):
    rng = np.random.default_rng(6100 + 16 * mode + fe)
    lens = [1, 3, 4, 5, 7, 8, 9, 31, 33, 124, 127, 128, 129, 132, 255, 256, 257, 300, 511, 513, 600]
    qs = W._make_set(rng, np.asarray(lens), np.full(4, 0.25))
    targets = []
    for k in range(len(lens)):   # long gaps on either side, so runs pass a warp's 32 cells
        c = W.mutate(rng, qs.seq(k), 0.04, 0.02)
        cut = len(c) // 2
        gap = int(rng.integers(0, 70))
        mid = rng.integers(0, 4, gap).astype(np.uint8)
        c = np.concatenate([c[:cut], mid, c[cut:]]) if k % 2 else np.concatenate([c[:cut], c[cut + min(gap, max(0, len(c) - cut - 1)):]])
        targets.append(np.concatenate([rng.integers(0, 4, 5).astype(np.uint8), c]).astype(np.uint8))
    db = W.SeqSet.from_list(targets)
    pairs = np.zeros(len(lens), W.PAIR_DTYPE)
    pairs["query_id"] = pairs["target_id"] = np.arange(len(lens))
    pairs["t_len"] = db.lengths
    S = W.dna_matrix(2, -3)
    r = ctx.align(ctx.load_set(db, 4), ctx.load_set(qs, 4), S, 3, 1, mode=mode, free_ends=fe, pairs=pairs)
    ctx.traceback(r)
    check_traceback(r.hits(), r.cigar(), qs, db, S, 3, 1, mode, fe)


@pytest.mark.parametrize("n", [1, 480])
@pytest.mark.parametrize("indels", [0.0, 0.08])
def test_long_walk_with_and_without_the_next_window(ctx, n, indels):
    """Few hits walk with the next band's window loaded ahead, many without;
    indels take the walk off the predicted diagonal."""
    rng = np.random.default_rng(6200 + n)
    q = rng.integers(0, 4, 5200).astype(np.uint8)
    t = W.mutate(rng, q, 0.1, indels, alphabet=4)
    Q = W.SeqSet.from_list([q])
    T = W.SeqSet.from_list([t])
    pairs = np.zeros(n, W.PAIR_DTYPE)
    pairs["t_len"] = len(t)
    res = ctx.align(ctx.load_set(T, 4), ctx.load_set(Q, 4), W.dna_matrix(2, -3), 5, 2, mode=dsa.GLOBAL, pairs=pairs)
    ctx.traceback(res)
    hits, cigar = res.hits(), res.cigar()
    for h in (hits[0], hits[-1]):
        ops = cigar[int(h["cigar_off"]):int(h["cigar_off"]) + int(h["cigar_len"])]
        i = j = score = 0
        for c in ops:
            length, op = int(c) >> 4, int(c) & 15
            if op == 0:
                score += int(np.where(q[i:i + length] == t[j:j + length], 2, -3).sum())
            else:
                score -= 5 + 2 * (length - 1)
            i += length if op in (0, 1) else 0
            j += length if op in (0, 2) else 0
        assert (i, j, score) == (len(q), len(t), int(h["score"]))
