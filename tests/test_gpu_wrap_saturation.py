"""Saturation on the wrapping forms of local search: queries and targets whose
scores leave the summed forms' range, so that values really pass 16 bits, beside
ordinary queries in the other half and over several bands, on the wavefronts and on
the inter-sequence kernel at both strip heights.  Scores, ends and the number of
reruns against the oracle."""
import numpy as np
import pytest

from paper_1701_01575_gb300 import dsa
from paper_1701_01575_gb300 import workloads as W

from test_gpu_parity import assert_same, gpu_all, oracle_all

pytestmark = pytest.mark.gpu

ROUTES = [("0", None), ("1000000", "28"), ("1000000", "20")]   # long threshold, inter-sequence rows


@pytest.fixture(scope="module")
def ctx():
    from paper_1701_01575_gb300 import build
    build.build()
    c = dsa.Context(0)
    yield c
    c.close()


def _route(monkeypatch, thr, rows):
    monkeypatch.setenv("DSA_LONG_THRESHOLD", thr)
    monkeypatch.setenv("DSA_AUTOTUNE", "off")
    if rows:
        monkeypatch.setenv("DSA_INTER_ROWS", rows)
    else:
        monkeypatch.delenv("DSA_INTER_ROWS", raising=False)


def _past_the_summed_range(smax, m, n, o, e):
    """Values with e j added, their bias and the last steps' margin need more than 16 bits."""
    return smax * min(m, n) + e * (n + 64) + (512 + o + 64 * e) + 2 * (o + e) + 512 >= 65536


@pytest.mark.parametrize("thr,rows", ROUTES)
def test_protein_runs(ctx, thr, rows, monkeypatch):
    _route(monkeypatch, thr, rows)
    rng = np.random.default_rng(8000)
    bg = W.protein_background()
    w = W.PROTEIN_LETTERS.index("W")
    runs = [np.full(n, w, np.uint8) for n in (6000, 2976, 2977, 2978, 2979, 3100)]
    queries = W.SeqSet.from_list(runs + [rng.choice(20, n, p=bg).astype(np.uint8) for n in (70, 500, 2500)])
    db = W.SeqSet.from_list(runs + [rng.choice(20, n, p=bg).astype(np.uint8) for n in (5, 33, 200, 3000)])
    S = W.blosum62()
    assert _past_the_summed_range(11, 6000, 6000, 11, 1)
    want = oracle_all(queries, db, S, 11, 1)
    got = gpu_all(ctx, queries, db, S, 11, 1)
    assert_same(got[:3], want, f"thr={thr} rows={rows}")
    assert want[0].max() > 65535 and got[4] == int((want[0] > 32767 - 11).sum())
    assert (got[5].phase_cells()["inter16"] == 0) == (thr == "0")


@pytest.mark.parametrize("thr,rows", ROUTES)
@pytest.mark.parametrize("pssm", [False, True])
def test_steep_scores(ctx, thr, rows, pssm, monkeypatch):
    """Matches of 40: short sequences reach the range, with gaps inside them."""
    _route(monkeypatch, thr, rows)
    rng = np.random.default_rng(8100)
    bg = np.full(4, 0.25)
    queries = W._make_set(rng, np.array([2000, 819, 820, 300, 40, 1500]), bg)
    targets = [W.mutate(rng, queries.seq(k), 0.01, 0.004) for k in range(queries.n)]
    targets += [queries.seq(1).copy(), queries.seq(2).copy()] + [rng.integers(0, 4, n).astype(np.uint8) for n in (1, 64, 900)]
    db = W.SeqSet.from_list(targets)
    S = np.full((4, 4), -30, np.int8)
    np.fill_diagonal(S, 40)
    assert _past_the_summed_range(40, 2000, int(db.lengths.max()), 50, 3)
    want = oracle_all(queries, db, S, 50, 3)
    if pssm:
        d, q = ctx.load_set(db, 4), ctx.load_set(queries, 4)
        r = ctx.align_pssm(d, q, S[queries.codes].astype(np.int8), 50, 3)
        h = r.hits()
        got = [h[f].reshape(queries.n, db.n) for f in ("score", "q_end", "t_end")]
        reruns = r.stats()[1]
    else:
        g = gpu_all(ctx, queries, db, S, 50, 3)
        got, reruns = g[:3], g[4]
    assert_same(got, want, f"thr={thr} rows={rows} pssm={pssm}")
    assert want[0].max() > 65535 and reruns == int((want[0] > 32767 - 40).sum()) > 3
