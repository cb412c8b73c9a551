"""After its first call on a device, in whatever mode, the allocation-free call
loads nothing more: in a process of its own, a global DNA call comes first, then
a local and a semi-global protein call (other kernels) are captured into a graph
with device memory use watched, and the replay gives what dsa_align gives."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r"""
import numpy as np, torch
from paper_1701_01575_gb300 import dsa, workloads as W

lib = dsa.load_library()
rng = np.random.default_rng(8100)

def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a).view(np.uint8).copy()).cuda()

def job(A, lens, S, o, e, mode, fe):
    bg = np.full(A, 1 / A)
    qs, db = W._make_set(rng, np.asarray(lens), bg), W._make_set(rng, rng.integers(1, 300, 30), bg)
    p = np.zeros(60, W.PAIR_DTYPE)
    p["query_id"], p["target_id"] = rng.integers(0, qs.n, 60), rng.integers(0, db.n, 60)
    p["t_len"] = db.lengths[p["target_id"]]
    bufs = [dev(x) for x in (qs.codes, qs.offsets, db.codes, db.offsets, p, S)]
    return dict(qs=qs, db=db, p=p, S=S, o=o, e=e, mode=mode, fe=fe, bufs=bufs,
                out=torch.full((3, 60), 12345, dtype=torch.int32, device="cuda"))

def call(j):
    b, out = j["bufs"], j["out"]
    rc = lib.dsa_score_pairs_noalloc(
        b[0].data_ptr(), b[1].data_ptr(), j["qs"].n, b[2].data_ptr(), b[3].data_ptr(), j["db"].n,
        b[4].data_ptr(), 60, j["mode"], j["fe"], b[5].data_ptr(), j["S"].shape[0], j["o"], j["e"], 300,
        out[0].data_ptr(), out[1].data_ptr(), out[2].data_ptr(), torch.cuda.current_stream().cuda_stream)
    assert rc == 0, (rc, lib.dsa_last_error())

first = job(4, [30, 90, 140], W.dna_matrix(2, -3), 5, 2, dsa.GLOBAL, 15)
rest = [job(24, [20, 130, 400], W.blosum62(), 11, 1, dsa.LOCAL, 15),
        job(24, [20, 130, 400], W.blosum62(), 11, 1, dsa.SEMIGLOBAL, 12),
        job(4, [20, 130, 400], W.dna_matrix(1, -4), 6, 1, dsa.LOCAL, 15)]
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):      # torch's own first capture
    rest[0]["out"].fill_(1)
call(first)
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    free = torch.cuda.mem_get_info()[0]
    for j in rest:
        call(j)
    assert torch.cuda.mem_get_info()[0] == free, "the captured calls took device memory"
graph.replay()
torch.cuda.synchronize()
ctx = dsa.Context(0)
for j in [first] + rest:
    A = j["S"].shape[0]
    h = ctx.align(ctx.load_set(j["db"], A), ctx.load_set(j["qs"], A), j["S"], j["o"], j["e"], mode=j["mode"],
                  free_ends=j["fe"], pairs=j["p"], flags=dsa.FORCE_INT32).hits()
    assert (j["out"].cpu().numpy() == np.stack([h["score"], h["q_end"], h["t_end"]])).all()
print("captured ok")
"""


def test_other_modes_under_capture_after_one_call():
    from paper_1701_01575_gb300 import build
    build.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, PYTHONPATH=root)
    r = subprocess.run([sys.executable, "-c", PROGRAM], cwd=root, env=env, capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0 and "captured ok" in r.stdout, r.stderr[-2000:]
