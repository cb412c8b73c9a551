"""The long-pair walk's CIGAR, with the next band's window loaded ahead (few hits)
and without (many), is the oracle's, word for word: indels and a long gap take the
walk off the diagonal that its window was placed on."""
import numpy as np
import pytest

import oracle
from paper_1701_01575_gb300 import dsa
from paper_1701_01575_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 480])
@pytest.mark.parametrize("mode", [dsa.GLOBAL, dsa.LOCAL])
def test_cigar_is_the_oracles(n, mode):
    from paper_1701_01575_gb300 import build
    build.build()
    rng = np.random.default_rng(8200 + mode)
    q = rng.integers(0, 4, 2600).astype(np.uint8)
    t = W.mutate(rng, q, 0.1, 0.05, alphabet=4)
    t = np.concatenate([t[:900], rng.integers(0, 4, 333).astype(np.uint8), t[900:]])   # more than a window's drift
    S, o, e = W.dna_matrix(2, -3), 5, 1
    ctx = dsa.Context(0)
    pairs = np.zeros(n, W.PAIR_DTYPE)
    pairs["t_len"] = len(t)
    assert len(q) * len(t) >= 4 << 20   # the band pipeline
    res = ctx.align(ctx.load_set(W.SeqSet.from_list([t]), 4), ctx.load_set(W.SeqSet.from_list([q]), 4), S, o, e,
                    mode=mode, pairs=pairs)
    ctx.traceback(res)
    hits, cigar = res.hits(), res.cigar()
    h = hits[0]
    qb, tb, want = oracle.traceback(q, t, S, o, e, mode, 15, int(h["q_end"]), int(h["t_end"]))
    for h in (hits[0], hits[-1], hits[n // 2]):
        got = cigar[int(h["cigar_off"]):int(h["cigar_off"]) + int(h["cigar_len"])]
        assert (int(h["q_begin"]), int(h["t_begin"])) == (qb, tb) and got.tolist() == want.tolist()
