"""The tuner keeps apart what its size bins alone would merge: searches whose
longest query and target take them to another kernel, and queries that fill
their strips differently."""
import json

import numpy as np
import pytest

from paper_1701_01575_gb300 import dsa
from paper_1701_01575_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,first,second", [
    (dsa.GLOBAL, [2900] * 3, [3000] * 3),      # 11 x 3,000 passes the summed form's range
    (dsa.LOCAL, [64] * 10, [80] * 8)])         # four strips of 16 and three of 28; five and three
def test_one_bin_two_entries(mode, first, second, tmp_path, monkeypatch):
    from paper_1701_01575_gb300 import build
    build.build()
    cache = tmp_path / "tune.json"
    monkeypatch.setenv("DSA_AUTOTUNE_CACHE", str(cache))
    for name in ("DSA_AUTOTUNE", "DSA_INTER_ROWS", "DSA_LONG_THRESHOLD"):
        monkeypatch.delenv(name, raising=False)
    rng = np.random.default_rng(7900 + mode)
    bg = W.protein_background()
    ctx = dsa.Context(0)
    d = ctx.load_set(W._make_set(rng, np.concatenate([rng.integers(50, 400, 300), [3100]]), bg), 24)
    seen = []
    for lengths in (first, second, first):
        q = ctx.load_set(W._make_set(rng, np.asarray(lengths), bg), 24)
        ctx.align(d, q, W.blosum62(), 11, 1, mode=mode, top_k=5).free()
        seen.append({k for k in json.loads(cache.read_text()) if k.endswith("|thr")})
    assert len(seen[0]) == 1 and len(seen[1]) == 2 and seen[2] == seen[1]
