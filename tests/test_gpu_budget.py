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
