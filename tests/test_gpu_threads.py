"""Host threads, each with a context of its own, that launch the same
kernels with different alphabets (so with different amounts of shared memory)
at the same time: every call succeeds and gives what it gives alone."""
import threading

import numpy as np
import pytest

from paper_1701_01575_gb300 import dsa
from paper_1701_01575_gb300 import workloads as W

pytestmark = pytest.mark.gpu

CALLS = 400


def _jobs(what, monkeypatch):
    """(alphabet, call) per thread; call(ctx, db, queries, pairs) -> arrays."""
    monkeypatch.setenv("DSA_LONG_THRESHOLD", "1000000" if what == "inter" else "0")
    monkeypatch.setenv("DSA_AUTOTUNE", "off")
    rng = np.random.default_rng(7100 + len(what))
    jobs = []
    for A in ((4, 24) if what != "pairs" else (12, 24)):
        bg = np.full(A, 1 / A)
        S = np.full((A, A), -2, np.int8)
        np.fill_diagonal(S, 5)
        # more queries than one band of 8-row strips holds: 24 rows, the largest profiles
        qs = W._make_set(rng, rng.integers(100, 170, 24), bg)
        db = W._make_set(rng, rng.integers(20, 60, 64), bg)
        pairs = np.zeros(400, W.PAIR_DTYPE)
        pairs["query_id"] = rng.integers(0, qs.n, len(pairs))
        pairs["target_id"] = rng.integers(0, db.n, len(pairs))
        pairs["t_len"] = db.lengths[pairs["target_id"]]
        jobs += [(A, S, qs, db, pairs)] * 2
    return jobs


@pytest.mark.parametrize("what", ["wave", "inter", "pairs"])
def test_calls_of_two_alphabets_at_once(what, monkeypatch):
    from paper_1701_01575_gb300 import build
    build.build()
    jobs = _jobs(what, monkeypatch)
    start = threading.Barrier(len(jobs))
    errors = []

    def worker(A, S, qs, db, pairs):
        try:
            ctx = dsa.Context(0)
            d, q = ctx.load_set(db, A), ctx.load_set(qs, A)
            kw = {"pairs": pairs} if what == "pairs" else {"top_k": 5}
            want = ctx.align(d, q, S, 7, 1, **kw).hits().copy()
            start.wait()
            for _ in range(CALLS):
                r = ctx.align(d, q, S, 7, 1, **kw)
                if not (r.hits() == want).all():
                    errors.append(f"A={A}: another result")
                    return
                r.free()
        except Exception as ex:   # reported by the test's own thread
            errors.append(f"A={A}: {ex!r}")
            start.abort()

    threads = [threading.Thread(target=worker, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
