"""Explicit pairs on the wavefront form (4 to 32 lanes a pair): scores and end
cells against the oracle at the edges of its blocks, groups and bands, in
every mode and set of free ends, and the rule that sends a pair there."""
import numpy as np
import pytest

import oracle
from paper_1701_01575_gb300 import dsa
from paper_1701_01575_gb300 import workloads as W

from test_gpu_parity import assert_same

pytestmark = pytest.mark.gpu

MODES = [(dsa.LOCAL, 15), (dsa.GLOBAL, 15), (dsa.SEMIGLOBAL, 15), (dsa.SEMIGLOBAL, 12),
         (dsa.SEMIGLOBAL, 3), (dsa.SEMIGLOBAL, 10), (dsa.SEMIGLOBAL, 5), (dsa.SEMIGLOBAL, 0)]
# query lengths around every group's rows (64 ... 1,024) and past one band
EDGES = [1, 2, 7, 8, 9, 12, 13, 63, 64, 65, 95, 96, 97, 127, 128, 129, 159, 160, 161, 191, 192, 193,
         255, 256, 257, 320, 321, 383, 384, 385, 512, 513, 640, 641, 768, 769, 1024, 1025, 1281, 1537, 2100]


@pytest.fixture(scope="module")
def ctx():
    from paper_1701_01575_gb300 import build
    build.build()
    c = dsa.Context(0)
    yield c
    c.close()


def _check(ctx, qs, db, pairs, S, o, e, mode, fe, what, flags=0):
    A = S.shape[0]
    r = ctx.align(ctx.load_set(db, A), ctx.load_set(qs, A), S, o, e, mode=mode, free_ends=fe,
                  pairs=pairs, flags=flags)
    h = r.hits()
    want = oracle.score_pairs(qs.codes, qs.offsets, db.codes, db.offsets, pairs["query_id"],
                              pairs["target_id"], S, o, e, mode, fe, pair_toff=pairs["t_offset"],
                              pair_tlen=pairs["t_len"])
    assert_same((h["score"], h["q_end"], h["t_end"]), want, what)
    return r


def _set(rng, lens, letters, probs):
    """Queries of the given lengths, each with windows of one residue, of its
    own mutated copy and of an unrelated stretch of a longer target."""
    qs = W._make_set(rng, np.asarray(lens), probs)
    targets, pairs = [], []
    for k, m in enumerate(lens):
        copy = W.mutate(rng, qs.seq(k), 0.1, 0.03, alphabet=letters)
        left, right = rng.integers(0, 40, 2)
        t = np.concatenate([rng.integers(0, letters, left), copy, rng.integers(0, letters, right + 3),
                            rng.integers(0, letters, 211)]).astype(np.uint8)
        targets.append(t)
        n = len(t)
        for off, length in ((0, n), (int(left), max(1, len(copy))), (n - 1, 1), (n - 200, int(rng.integers(2, 200)))):
            pairs.append((k, k, off, length))
    arr = np.zeros(len(pairs), W.PAIR_DTYPE)
    for x, (q, t, off, length) in enumerate(pairs):
        arr[x] = (q, t, off, length, 0)
    return qs, W.SeqSet.from_list(targets), arr[rng.permutation(len(arr))]


@pytest.mark.parametrize("mode,fe", MODES)
@pytest.mark.parametrize("alphabet", ["protein", "dna"])
def test_block_and_band_edges(ctx, alphabet, mode, fe):
    rng = np.random.default_rng(3100 + 16 * mode + fe + (alphabet == "dna"))
    if alphabet == "protein":
        qs, db, pairs = _set(rng, EDGES, 20, W.protein_background())
        S, o, e = W.blosum62(), 11, 1
    else:
        qs, db, pairs = _set(rng, EDGES, 4, np.full(4, 0.25))
        S, o, e = W.dna_matrix(2, -3), 5, 2
    r = _check(ctx, qs, db, pairs, S, o, e, mode, fe, f"{alphabet} mode={mode} fe={fe}")
    assert r.phase_cells()["int32"] == 0


@pytest.mark.parametrize("o,e", [(1, 0), (3, 3), (20, 9), (90, 2)])
@pytest.mark.parametrize("mode,fe", [(dsa.LOCAL, 15), (dsa.GLOBAL, 15), (dsa.SEMIGLOBAL, 9)])
def test_gap_costs(ctx, o, e, mode, fe):
    """Gap costs at the edges of the byte tables, an asymmetric matrix over an
    odd alphabet."""
    rng = np.random.default_rng(3200 + o + e + mode)
    S = rng.integers(-9, 12, (7, 7)).astype(np.int8)
    qs, db, pairs = _set(rng, [1, 40, 64, 100, 129, 300, 777, 1100], 7, np.full(7, 1 / 7))
    _check(ctx, qs, db, pairs, S, o, e, mode, fe, f"o={o} e={e} mode={mode}")


@pytest.mark.parametrize("mode,fe", [(dsa.LOCAL, 15), (dsa.GLOBAL, 15), (dsa.SEMIGLOBAL, 15)])
def test_range_rule_and_rerun(ctx, mode, fe):
    """Pairs on both sides of the 16-bit rule among ordinary ones: local scores
    past 32767 are rerun, global ones past the rule take the int32 kernel."""
    rng = np.random.default_rng(3300 + mode)
    S = np.full((5, 5), -7, np.int8)
    np.fill_diagonal(S, 40)
    lens = [1500, 1600, 815, 821, 30, 200, 2000]
    qs = W._make_set(rng, np.asarray(lens), np.full(5, 0.2))
    db = W.SeqSet.from_list([qs.seq(k).copy() for k in range(len(lens))])
    pairs = np.zeros(len(lens), W.PAIR_DTYPE)
    pairs["query_id"] = pairs["target_id"] = np.arange(len(lens))
    pairs["t_len"] = lens
    r = _check(ctx, qs, db, pairs, S, 20, 3, mode, fe, f"range mode={mode}")
    if mode == dsa.LOCAL:
        assert r.stats()[1] == sum(40 * n > 32767 - 40 for n in lens)
    else:
        assert r.stats()[1] == 0 and 0 < r.phase_cells()["int32"] < r.stats()[0]


@pytest.mark.parametrize("mode,fe", [(dsa.LOCAL, 15), (dsa.GLOBAL, 15), (dsa.SEMIGLOBAL, 12)])
@pytest.mark.parametrize("alphabet", ["dna", "protein"])
def test_many_pairs_take_two_lanes_each(ctx, alphabet, mode, fe):
    """Enough pairs for the densest classes (two lanes a pair)."""
    rng = np.random.default_rng(3500 + mode + len(alphabet))
    bg = np.full(4, 0.25) if alphabet == "dna" else W.protein_background()
    S, o, e = (W.dna_matrix(1, -4), 6, 1) if alphabet == "dna" else (W.blosum62(), 11, 1)
    qs = W._make_set(rng, rng.integers(1, 90, 400), bg)
    db = W._make_set(rng, rng.integers(1, 60, 300), bg)
    pairs = np.zeros(33_000, W.PAIR_DTYPE)
    pairs["query_id"] = rng.integers(0, qs.n, len(pairs))
    pairs["target_id"] = rng.integers(0, db.n, len(pairs))
    pairs["t_len"] = db.lengths[pairs["target_id"]]
    _check(ctx, qs, db, pairs, S, o, e, mode, fe, f"dense {alphabet} mode={mode}")


@pytest.mark.parametrize("mode,fe", [(dsa.LOCAL, 15), (dsa.SEMIGLOBAL, 12)])
def test_long_pairs_among_short_ones(ctx, mode, fe):
    """A call that also holds pairs of the band pipeline, on the device and on
    the host, and the same pairs on the int32 kernel."""
    import torch
    rng = np.random.default_rng(3400 + mode)
    lens = [2100, 50, 700, 2500, 128, 33, 1000] * 3
    qs = W._make_set(rng, np.asarray(lens), np.full(4, 0.25))
    db = W.SeqSet.from_list([W.mutate(rng, qs.seq(k), 0.05, 0.02) for k in range(len(lens))])
    pairs = np.zeros(len(lens), W.PAIR_DTYPE)
    pairs["query_id"] = pairs["target_id"] = np.arange(len(lens))
    pairs["t_len"] = db.lengths
    S = W.dna_matrix(2, -3)
    r = _check(ctx, qs, db, pairs, S, 5, 2, mode, fe, f"mixed mode={mode}")
    assert 0 < r.phase_cells()["intra16"] < r.stats()[0]
    ref = r.hits()
    on_dev = torch.from_numpy(pairs.view(np.uint8)).cuda()
    d, q = ctx.load_set(db, 4), ctx.load_set(qs, 4)
    assert (ctx.align(d, q, S, 5, 2, mode=mode, free_ends=fe, pairs=on_dev).hits() == ref).all()
    _check(ctx, qs, db, pairs, S, 5, 2, mode, fe, "int32", flags=dsa.FORCE_INT32)
