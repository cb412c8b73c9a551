"""Database search with every target on the wavefront kernel: scores and end
cells against the oracle at the edges of its strips (16 and 24 rows), lane
groups and bands, in its three forms, with targets of one residue to thousands
and query streams of unequal halves."""
import numpy as np
import pytest

from paper_1701_01575_gb300 import dsa
from paper_1701_01575_gb300 import workloads as W

from test_gpu_parity import assert_same, gpu_all, oracle_all

pytestmark = pytest.mark.gpu

MODES = [(dsa.LOCAL, 15), (dsa.GLOBAL, 15), (dsa.SEMIGLOBAL, 15), (dsa.SEMIGLOBAL, 12),
         (dsa.SEMIGLOBAL, 3), (dsa.SEMIGLOBAL, 10), (dsa.SEMIGLOBAL, 5)]
QUERIES = {
    "one": [300],                                           # an empty high half
    "short": [1, 2, 15, 16, 17, 23, 24, 25, 31, 32, 33, 47, 48, 49, 64, 96],
    "bands": [24 * 8, 24 * 8 + 1, 24 * 16 - 1, 24 * 32 + 5, 700, 1200, 5, 130],
}


@pytest.fixture(scope="module")
def ctx():
    from paper_1701_01575_gb300 import build
    build.build()
    c = dsa.Context(0)
    yield c
    c.close()


def _db(rng, queries, bg, longest):
    lens = np.concatenate([[1, 2, 3, 4, 5, 7, 8, 31, 32, 33, longest], rng.integers(1, 400, 120)])
    seqs = [rng.choice(len(bg), int(n), p=bg).astype(np.uint8) for n in lens]
    for k in range(queries.n):   # a mutated copy of each query inside a target
        copy = W.mutate(rng, queries.seq(k), 0.2, 0.03, alphabet=len(bg))
        seqs.append(np.concatenate([rng.choice(len(bg), 9, p=bg).astype(np.uint8), copy]))
    return W.SeqSet.from_list(seqs)


@pytest.mark.parametrize("which", list(QUERIES))
@pytest.mark.parametrize("mode,fe", MODES)
def test_strip_group_and_band_edges(ctx, which, mode, fe, monkeypatch):
    monkeypatch.setenv("DSA_LONG_THRESHOLD", "0")
    rng = np.random.default_rng(5100 + 16 * mode + fe + len(which))
    bg = W.protein_background()
    queries = W._make_set(rng, np.asarray(QUERIES[which]), bg)
    db = _db(rng, queries, bg, 2600)
    S = W.blosum62()
    g = gpu_all(ctx, queries, db, S, 11, 1, mode=mode, fe=fe)
    assert_same(g[:3], oracle_all(queries, db, S, 11, 1, mode, fe), f"{which} mode={mode} fe={fe}")
    assert g[4] == 0 and g[5].phase_cells()["inter16"] == 0


@pytest.mark.parametrize("o,e", [(1, 0), (3, 3), (60, 40), (500, 300)])
@pytest.mark.parametrize("mode,fe", [(dsa.LOCAL, 15), (dsa.GLOBAL, 15), (dsa.SEMIGLOBAL, 6)])
def test_gap_costs_of_every_form(ctx, o, e, mode, fe, monkeypatch):
    """Small alphabets force ties; large costs leave the summed forms' range
    (local: the wrapping form, global: the kernels with a range flag)."""
    monkeypatch.setenv("DSA_LONG_THRESHOLD", "0")
    rng = np.random.default_rng(5200 + o + mode)
    bg = np.full(4, 0.25)
    queries = W._make_set(rng, np.array([40, 260, 33, 100, 17]), bg)
    db = _db(rng, queries, bg, 900)
    S = W.dna_matrix(2, -3)
    g = gpu_all(ctx, queries, db, S, o, e, mode=mode, fe=fe)
    assert_same(g[:3], oracle_all(queries, db, S, o, e, mode, fe), f"o={o} e={e} mode={mode}")


def test_saturated_pairs_are_flagged_and_rerun(ctx, monkeypatch):
    """Bests on both sides of the 16-bit rule, beside ordinary queries in the
    other half and in the same stream."""
    monkeypatch.setenv("DSA_LONG_THRESHOLD", "0")
    rng = np.random.default_rng(5300)
    w = W.PROTEIN_LETTERS.index("W")
    bg = W.protein_background()
    seqs = [np.full(n, w, np.uint8) for n in (2976, 2978, 3300)]
    queries = W.SeqSet.from_list(seqs + [rng.choice(20, n, p=bg).astype(np.uint8) for n in (70, 500)])
    db = W.SeqSet.from_list(seqs + [rng.choice(20, n, p=bg).astype(np.uint8) for n in (5, 200, 3000)])
    S = W.blosum62()
    orc = oracle_all(queries, db, S, 11, 1)
    g = gpu_all(ctx, queries, db, S, 11, 1)
    assert_same(g[:3], orc, "saturated")
    assert g[4] == int((orc[0] > 32767 - 11).sum()) > 0


def test_modelled_threshold_matches_the_wavefronts(ctx, monkeypatch):
    """Without a tuned or forced threshold, a database for both kernels."""
    monkeypatch.setenv("DSA_AUTOTUNE", "off")
    monkeypatch.delenv("DSA_LONG_THRESHOLD", raising=False)
    rng = np.random.default_rng(5400)
    bg = W.protein_background()
    queries = W._make_set(rng, np.array([30, 90]), bg)
    db = W._make_set(rng, np.concatenate([W.lognormal_int(rng, 300, 0.7, 5000, 60000)]), bg)
    S = W.blosum62()
    a = ctx.align(ctx.load_set(db, 24), ctx.load_set(queries, 24), S, 11, 1)
    monkeypatch.setenv("DSA_LONG_THRESHOLD", "0")
    b = ctx.align(ctx.load_set(db, 24), ctx.load_set(queries, 24), S, 11, 1)
    assert (a.hits() == b.hits()).all()


@pytest.mark.parametrize("lengths", [[1], [8], [9], [255], [256], [256, 256], [1, 7, 8, 9, 15, 16, 17, 64, 65, 100],
                                     [250, 3, 3, 120, 100, 31]])
@pytest.mark.parametrize("mode,fe", [(dsa.LOCAL, 15), (dsa.GLOBAL, 15), (dsa.SEMIGLOBAL, 6)])
def test_short_strips_of_small_searches(ctx, lengths, mode, fe, monkeypatch):
    """Queries that fill one band at 8 rows at most."""
    monkeypatch.setenv("DSA_LONG_THRESHOLD", "0")
    rng = np.random.default_rng(5500 + sum(lengths) + mode)
    bg = W.protein_background()
    queries = W._make_set(rng, np.asarray(lengths), bg)
    db = _db(rng, queries, bg, 700)
    S = W.blosum62()
    g = gpu_all(ctx, queries, db, S, 11, 1, mode=mode, fe=fe)
    assert_same(g[:3], oracle_all(queries, db, S, 11, 1, mode, fe), f"{lengths} mode={mode}")
    assert g[5].phase_cells()["inter16"] == 0


@pytest.mark.parametrize("lengths", [[100], [176], [300], [24 * 16 + 1], [700, 30, 100], [1100, 16, 17, 3]])
@pytest.mark.parametrize("mode,fe", MODES)
@pytest.mark.parametrize("n_targets", [24000, 24001])
def test_two_targets_a_lane(ctx, lengths, mode, fe, n_targets, monkeypatch):
    """Queries whose streams would leave one half idle (one of them, or one much
    longer than the rest) against enough targets that the work outlasts the
    longest one's chain: strips of 8 (100), 16 (176) and 24 rows, even and odd
    numbers of targets; by matrix and, in local mode, as a profile."""
    monkeypatch.setenv("DSA_LONG_THRESHOLD", "0")
    rng = np.random.default_rng(5600 + sum(lengths) + 16 * mode + fe)
    bg = W.protein_background()
    queries = W._make_set(rng, np.asarray(lengths), bg)
    lens = rng.integers(1, 100, n_targets)
    lens[:4] = (100, 1, 2, 130) if sum(lengths) < 1000 else (900, 1, 500, 300)
    assert max(lengths) * 2 * 10 > sum(lengths) * 12
    rows = 8 if max(lengths) <= 100 else 24
    assert (max(lengths) // rows) * int(lens.sum()) * 4 >= 3 * int(lens.max()) * 152 * 512
    db = W._make_set(rng, lens, bg)
    for k, n in enumerate(lengths):   # a mutated piece of each query inside a target
        at = int(db.offsets[3 + 5 * k])
        room = int(db.offsets[4 + 5 * k]) - at
        piece = W.mutate(rng, queries.seq(k), 0.2, 0.02, alphabet=len(bg))[:room]
        db.codes[at:at + len(piece)] = piece
    S = W.blosum62()
    for o, e in ((11, 1), (2, 1)):   # the profile's bytes as they are; lifted to 0 or more
        g = gpu_all(ctx, queries, db, S, o, e, mode=mode, fe=fe)
        assert_same(g[:3], oracle_all(queries, db, S, o, e, mode, fe), f"{lengths} mode={mode} o={o}")
        assert g[5].phase_cells()["inter16"] == 0
    if mode == dsa.LOCAL:
        d, q = ctx.load_set(db, 24), ctx.load_set(queries, 24)
        a = ctx.align(d, q, S, 11, 1, top_k=50)
        b = ctx.align_pssm(d, q, S[queries.codes].astype(np.int8), 11, 1, top_k=50)
        assert (a.hits() == b.hits()).all()
