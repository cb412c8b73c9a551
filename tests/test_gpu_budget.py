"""Searches under a memory budget: what a call takes and gives back, and what
fits."""
import numpy as np
import pytest

from paper_1701_01575_gb300 import dsa
from paper_1701_01575_gb300 import workloads as W

from test_gpu_parity import assert_same, oracle_all

pytestmark = pytest.mark.gpu

MB = 1 << 20


def _hits(ctx, db, qs, S, o, e, A, **kw):
    r = ctx.align(ctx.load_set(db, A), ctx.load_set(qs, A), S, o, e, **kw)
    h = r.hits().copy()
    r.free()
    return h


def test_call_refused_beside_running_wavefronts(monkeypatch):
    """The long targets' wavefronts are running on the second stream when the
    boundary rows of the rest do not fit: the call fails, gives back what it
    took, and the calls after it are exact."""
    monkeypatch.setenv("DSA_AUTOTUNE", "off")
    rng = np.random.default_rng(7200)
    bg = W.protein_background()
    qs = W._make_set(rng, np.array([2000, 2000]), bg)
    db = W._make_set(rng, np.concatenate([np.full(100, 2500), rng.integers(100, 281, 60_000)]), bg)
    S = W.blosum62()
    big = dsa.Context(0)
    monkeypatch.setenv("DSA_LONG_THRESHOLD", "0")
    want = _hits(big, db, qs, S, 11, 1, 24, top_k=40)
    ctx = dsa.Context(0, mem_budget=90 * MB)
    d, q = ctx.load_set(db, 24), ctx.load_set(qs, 24)
    for _ in range(3):
        monkeypatch.setenv("DSA_LONG_THRESHOLD", "0")
        r = ctx.align(d, q, S, 11, 1, top_k=40)
        assert (r.hits() == want).all()
        r.free()
        held = ctx.mem_in_use()
        monkeypatch.setenv("DSA_LONG_THRESHOLD", "300")
        with pytest.raises(dsa.DsaError) as err:
            ctx.align(d, q, S, 11, 1, top_k=40)
        assert err.value.code == dsa.ERR_OVER_BUDGET and ctx.mem_in_use() == held
    ctx.sync()


@pytest.mark.parametrize("lens,budget", [([60_000] * 100, 80), ([300_000] + [200] * 3000, 200)])
def test_boundary_rows_follow_the_targets(lens, budget, monkeypatch):
    """Wavefronts of several bands: a few long targets, and one very long one
    among many short, take about a boundary row per target, not one of the
    longest for every warp of the chip."""
    monkeypatch.setenv("DSA_AUTOTUNE", "off")
    monkeypatch.setenv("DSA_LONG_THRESHOLD", "0")
    rng = np.random.default_rng(7300 + budget)
    bg = W.protein_background()
    qs = W._make_set(rng, np.array([2000]), bg)
    db = W._make_set(rng, np.array(lens), bg)
    S = W.blosum62()
    h = _hits(dsa.Context(0, mem_budget=budget * MB), db, qs, S, 11, 1, 24)
    assert_same((h["score"].reshape(1, -1), h["q_end"].reshape(1, -1), h["t_end"].reshape(1, -1)),
                oracle_all(qs, db, S, 11, 1), f"budget {budget} MB")


@pytest.mark.parametrize("mode", [dsa.LOCAL, dsa.GLOBAL, dsa.SEMIGLOBAL])
def test_more_items_than_slots(mode, monkeypatch):
    """Units of several bands whose items outnumber the resident CTAs, long
    targets in every unit: each CTA's boundary rows hold whatever it is dealt."""
    monkeypatch.setenv("DSA_AUTOTUNE", "off")
    rng = np.random.default_rng(7400 + mode)
    bg = W.protein_background()
    qs = W._make_set(rng, rng.integers(400, 1000, 24), bg)
    db = W._make_set(rng, np.concatenate([rng.integers(2000, 5000, 200), rng.integers(20, 700, 8000)]), bg)
    S = W.blosum62()
    ctx = dsa.Context(0)
    got = []
    for thr in ("0", "1000000"):
        monkeypatch.setenv("DSA_LONG_THRESHOLD", thr)
        got.append(_hits(ctx, db, qs, S, 11, 1, 24, mode=mode))
    assert (got[0] == got[1]).all()


def test_threshold_fits_the_budget(monkeypatch):
    """Many short queries against long targets, where the model would keep
    targets of some 13,000 residues on the inter-sequence kernel: 8 GB of
    boundary rows, which a small budget does not hold."""
    monkeypatch.setenv("DSA_AUTOTUNE", "off")
    monkeypatch.delenv("DSA_LONG_THRESHOLD", raising=False)
    rng = np.random.default_rng(7500)
    bg = np.full(4, 0.25)
    qs = W._make_set(rng, np.full(512, 60), bg)
    db = W._make_set(rng, rng.integers(2000, 20_000, 1500), bg)
    S = W.dna_matrix(2, -3)
    got = [_hits(dsa.Context(0, mem_budget=b), db, qs, S, 5, 2, 4, top_k=5) for b in (3 << 30, 0)]
    assert (got[0] == got[1]).all()
