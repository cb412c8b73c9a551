"""Search wavefronts of several bands on strips of 16 rows, whose boundary row
lanes read a block of four columns ahead: targets around those blocks, lane
groups with and without a target, one query stream and two."""
import numpy as np
import pytest

from paper_1701_01575_gb300 import dsa
from paper_1701_01575_gb300 import workloads as W

from test_gpu_parity import assert_same, gpu_all, oracle_all

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1701_01575_gb300 import build
    build.build()
    c = dsa.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("lengths", [[175] * 24, [64] * 40, [16] * 90 + [300], [1000], [1020, 990], [400] * 8])
@pytest.mark.parametrize("mode,fe", [(dsa.GLOBAL, 15), (dsa.SEMIGLOBAL, 15), (dsa.SEMIGLOBAL, 10), (dsa.LOCAL, 15)])
@pytest.mark.parametrize("n_targets", [37, 2500])
def test_bands_of_short_strips(ctx, lengths, mode, fe, n_targets, monkeypatch):
    monkeypatch.setenv("DSA_LONG_THRESHOLD", "0")
    rng = np.random.default_rng(7600 + sum(lengths) + 16 * mode + fe + n_targets)
    bg = W.protein_background()
    queries = W._make_set(rng, np.asarray(lengths), bg)
    lens = np.concatenate([[1, 2, 3, 4, 5, 7, 8, 9, 12, 13, 31, 32, 33], rng.integers(1, 90, n_targets - 14), [2300]])
    db = W._make_set(rng, lens, bg)
    at = int(db.offsets[-2])   # a related target
    piece = W.mutate(rng, queries.seq(0), 0.2, 0.02, alphabet=len(bg))[:2300]
    db.codes[at:at + len(piece)] = piece
    S = W.blosum62()
    g = gpu_all(ctx, queries, db, S, 11, 1, mode=mode, fe=fe)
    assert_same(g[:3], oracle_all(queries, db, S, 11, 1, mode, fe), f"{lengths[:2]} mode={mode} fe={fe}")
    assert g[5].phase_cells()["inter16"] == 0
