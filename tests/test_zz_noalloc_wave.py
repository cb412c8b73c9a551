"""The allocation-free scores on both of their kernels: pairs the wavefront
kernel takes (every mode, few pairs and many, queries of several bands), pairs
it leaves to the int32 kernel (scores past 16 bits, a matrix past its byte
tables) and pairs out of range among valid ones, against dsa_align."""
import numpy as np
import pytest

from paper_1701_01575_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(qs, db, pairs, mode, fe, S, o, e):
    import torch
    from paper_1701_01575_gb300 import build, dsa
    build.build()
    lib = dsa.load_library()

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).copy()).cuda()

    qc, qo, tc, to = dev(qs.codes), dev(qs.offsets), dev(db.codes), dev(db.offsets)
    dp, dm = dev(pairs), dev(S)
    n = len(pairs)
    out = torch.full((3, n), 12345, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    rc = lib.dsa_score_pairs_noalloc(qc.data_ptr(), qo.data_ptr(), qs.n, tc.data_ptr(), to.data_ptr(), db.n,
                                     dp.data_ptr(), n, mode, fe, dm.data_ptr(), S.shape[0], o, e,
                                     int(pairs["t_len"].max()), out[0].data_ptr(), out[1].data_ptr(),
                                     out[2].data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert rc == 0, lib.dsa_last_error()
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _want(qs, db, pairs, mode, fe, S, o, e):
    from paper_1701_01575_gb300 import dsa
    ctx = dsa.Context(0)
    try:
        A = S.shape[0]
        h = ctx.align(ctx.load_set(db, A), ctx.load_set(qs, A), S, o, e, mode=mode, free_ends=fe, pairs=pairs,
                      flags=dsa.FORCE_INT32).hits()
        return np.stack([h["score"], h["q_end"], h["t_end"]])
    finally:
        ctx.close()


def _pairs(rng, qs, db, n):
    p = np.zeros(n, W.PAIR_DTYPE)
    p["query_id"] = rng.integers(0, qs.n, n)
    p["target_id"] = rng.integers(0, db.n, n)
    tl = db.lengths[p["target_id"]]
    p["t_len"] = np.maximum(1, (rng.random(n) * tl).astype(np.int64))
    p["t_offset"] = (rng.random(n) * (tl - p["t_len"] + 1)).astype(np.int64)
    return p


@pytest.mark.parametrize("n_pairs", [1, 7, 500, 9001])
@pytest.mark.parametrize("mode,fe", [(0, 15), (1, 15), (2, 15), (2, 12), (2, 6)])
def test_every_mode_few_and_many_pairs(n_pairs, mode, fe):
    rng = np.random.default_rng(4100 + n_pairs + 16 * mode + fe)
    if n_pairs % 2:
        qs = W._make_set(rng, rng.integers(1, 400, 50), np.full(4, 0.25))
        db = W._make_set(rng, rng.integers(1, 700, 40), np.full(4, 0.25))
        S, o, e = W.dna_matrix(1, -4), 6, 1
    else:
        bg = W.protein_background()
        qs = W._make_set(rng, np.concatenate([[1, 64, 127, 128, 129, 256, 257, 513, 1025, 1300], rng.integers(1, 300, 40)]), bg)
        db = W._make_set(rng, rng.integers(1, 500, 60), bg)
        S, o, e = W.blosum62(), 11, 1
    p = _pairs(rng, qs, db, n_pairs)
    got, want = _run(qs, db, p, mode, fe, S, o, e), _want(qs, db, p, mode, fe, S, o, e)
    assert (got == want).all(), np.argwhere(got != want)[:5]


@pytest.mark.parametrize("mode", [0, 1, 2])
@pytest.mark.parametrize("what", ["scores", "tables"])
def test_pairs_left_to_int32(what, mode):
    """Scores past 16 bits for some pairs; a scoring whose tables pass a byte."""
    rng = np.random.default_rng(4200 + mode)
    S = np.full((4, 4), -5, np.int8)
    np.fill_diagonal(S, 40)
    o, e = (30, 2) if what == "scores" else (100, 60)
    qs = W._make_set(rng, np.array([1700, 900, 100, 30]), np.full(4, 0.25))
    db = W.SeqSet.from_list([qs.seq(k).copy() for k in range(4)])
    p = _pairs(rng, qs, db, 40)
    p["target_id"][:8] = p["query_id"][:8] = np.arange(8) % 4
    p["t_offset"][:8] = 0
    p["t_len"][:8] = db.lengths[np.arange(8) % 4]
    tl = db.lengths[p["target_id"]].astype(np.int64)
    p["t_len"] = np.minimum(p["t_len"], tl - p["t_offset"].astype(np.int64))
    got, want = _run(qs, db, p, mode, 15, S, o, e), _want(qs, db, p, mode, 15, S, o, e)
    assert want[0].max() > 32767
    assert (got == want).all(), np.argwhere(got != want)[:5]


def test_pairs_out_of_range_among_valid_ones():
    rng = np.random.default_rng(4300)
    qs = W._make_set(rng, rng.integers(1, 200, 30), np.full(4, 0.25))
    db = W._make_set(rng, rng.integers(20, 300, 20), np.full(4, 0.25))
    S = W.dna_matrix(2, -3)
    p = _pairs(rng, qs, db, 100)
    want = _want(qs, db, p, 2, 12, S, 5, 2)
    bad_code = int(p["query_id"][3])
    qs.codes[int(qs.offsets[bad_code])] = 9          # a code past the alphabet
    p["query_id"][10] = qs.n
    p["target_id"][20] = db.n
    p["t_offset"][30] = db.lengths[p["target_id"][30]]
    got = _run(qs, db, p, 2, 12, S, 5, 2)
    bad = np.isin(np.arange(100), [10, 20, 30]) | (p["query_id"] == bad_code)
    assert (got[:, bad] == np.array([[np.iinfo(np.int32).min], [-2], [-2]])).all()
    assert (got[:, ~bad] == want[:, ~bad]).all()
