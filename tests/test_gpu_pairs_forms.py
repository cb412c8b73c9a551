"""Which packed form a call's explicit pairs take, and that its results are the
oracle's: reads whose wavefront class is a quarter padding go to the per-thread
form (its row tuner then leaves an entry in the cache file), others stay on
the wavefronts, under DSA_AUTOTUNE=retune too."""
import json

import numpy as np
import pytest

import oracle
from paper_1701_01575_gb300 import dsa
from paper_1701_01575_gb300 import workloads as W

from test_gpu_parity import assert_same

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_1701_01575_gb300 import build
    build.build()
    c = dsa.Context(0)
    yield c
    c.close()


def _reads(rng, n, m, window):
    genome = rng.integers(0, 4, 300_000).astype(np.uint8)
    start = rng.integers(0, len(genome) - window - m, n)
    codes = genome[(start + max(0, (window - m) // 2))[:, None] + np.arange(m)]
    codes = np.where(rng.random(codes.shape) < 0.02, (codes + 1) % 4, codes).astype(np.uint8)
    p = np.zeros(n, W.PAIR_DTYPE)
    p["query_id"], p["t_offset"], p["t_len"] = np.arange(n), start, window
    return W.SeqSet(codes.reshape(-1), np.arange(n + 1, dtype=np.uint64) * np.uint64(m)), W.SeqSet.from_list([genome]), p


@pytest.mark.parametrize("mode,fe,m,window,n,per_thread", [
    (dsa.LOCAL, 15, 161, 170, 150_000, True), (dsa.LOCAL, 15, 98, 110, 300_000, True),
    (dsa.SEMIGLOBAL, 12, 193, 210, 200_000, True), (dsa.GLOBAL, 15, 325, 325, 200_000, True),
    (dsa.LOCAL, 15, 150, 160, 100_000, False), (dsa.SEMIGLOBAL, 12, 125, 140, 100_000, False),
    (dsa.LOCAL, 15, 161, 170, 4000, False)])
def test_form_and_results(ctx, mode, fe, m, window, n, per_thread, tmp_path, monkeypatch):
    cache = tmp_path / "tune.json"
    monkeypatch.setenv("DSA_AUTOTUNE_CACHE", str(cache))
    monkeypatch.delenv("DSA_AUTOTUNE", raising=False)
    monkeypatch.delenv("DSA_PAIRS_ROWS", raising=False)
    qs, db, pairs = _reads(np.random.default_rng(7700 + m + mode), n, m, window)
    S = W.dna_matrix(1, -4)
    r = ctx.align(ctx.load_set(db, 4), ctx.load_set(qs, 4), S, 6, 1, mode=mode, free_ends=fe, pairs=pairs)
    h = r.hits()
    want = oracle.score_pairs(qs.codes, qs.offsets, db.codes, db.offsets, pairs["query_id"], pairs["target_id"],
                              S, 6, 1, mode, fe, pair_toff=pairs["t_offset"], pair_tlen=pairs["t_len"])
    assert_same((h["score"], h["q_end"], h["t_end"]), want, f"m={m} mode={mode}")
    keys = json.loads(cache.read_text()) if cache.exists() else {}
    assert any("|pairs|" in k for k in keys) == per_thread


@pytest.mark.parametrize("mode", [dsa.LOCAL, dsa.GLOBAL])
def test_retuning_keeps_the_form(ctx, mode, tmp_path, monkeypatch):
    """Protein pairs past the per-thread form's narrow range: on the wavefronts
    under DSA_AUTOTUNE=retune as without it, none in int32."""
    monkeypatch.setenv("DSA_AUTOTUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.delenv("DSA_PAIRS_ROWS", raising=False)
    rng = np.random.default_rng(7800 + mode)
    bg = W.protein_background()
    qs = W._make_set(rng, rng.integers(50, 1200, 60), bg)
    db = W._make_set(rng, rng.integers(50, 1200, 90), bg)
    pairs = np.zeros(500, W.PAIR_DTYPE)
    pairs["query_id"], pairs["target_id"] = rng.integers(0, qs.n, 500), rng.integers(0, db.n, 500)
    pairs["t_len"] = db.lengths[pairs["target_id"]]
    S = W.blosum62()
    d, q = ctx.load_set(db, 24), ctx.load_set(qs, 24)
    launches, hits = [], []
    for tune in ("off", "retune"):
        monkeypatch.setenv("DSA_AUTOTUNE", tune)
        before = ctx.kernel_launches()
        r = ctx.align(d, q, S, 11, 1, mode=mode, pairs=pairs)
        hits.append(r.hits().copy())
        launches.append(ctx.kernel_launches() - before)
        assert r.phase_cells()["int32"] == 0 and r.phase_cells()["inter16"] > 0
    assert (hits[0] == hits[1]).all() and launches[0] == launches[1]
