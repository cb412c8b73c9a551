"""What users of this library have it do, as cases to be timed.

Every case goes through the public entry points of ``paper_1701_01575_gb300.dsa``
(or, for the allocation-free call, the C entry point itself).  Inputs are drawn
from a seed with the shapes of ``paper_1701_01575_gb300/workloads.py``; lengths
are the quantiles of their distribution in an order drawn from the seed, so a
case's cell count does not depend on the seed.
"""
import math

import numpy as np
import torch

from paper_1701_01575_gb300 import dsa, workloads

MODES = {"local": dsa.LOCAL, "global": dsa.GLOBAL, "semi": dsa.SEMIGLOBAL}
PROTEIN = (11, 1)        # BLOSUM62 gap open / extend of the protein workloads
READ = (1, -4, 6, 1)     # match, mismatch, open, extend of the read workloads
LONG = (2, -3, 5, 2)     # the same of the long DNA pairs
WINDOW_ENDS = dsa.FREE_T_BEGIN | dsa.FREE_T_END


def listed():
    return [
        # One protein against a small family or genome database: the smallest
        # search a user runs interactively; launches and host work count.
        {"name": "search_one", "kind": "search", "mode": "local", "queries": 1, "qlo": 128, "qhi": 128,
         "targets": 2000, "tlo": 50, "thi": 500, "top_k": 10, "host_queries": True},
        # The batched protein search of a whole reference database.
        {"name": "search_batch", "kind": "search", "mode": "local", "queries": 32, "qlo": 64, "qhi": 5000,
         "targets": 500_000, "tlo": 0, "thi": 0, "top_k": 10, "host_queries": False},
        # Semi-global search (whole query somewhere in the target, or the
        # reverse) of a mid-sized database, an odd number of queries.
        {"name": "search_semi", "kind": "search", "mode": "semi", "queries": 7, "qlo": 90, "qhi": 1100,
         "targets": 50_011, "tlo": 0, "thi": 0, "top_k": 10, "host_queries": False},
        # Profile (PSSM) search, as the inner step of an iterated search.
        {"name": "search_profile", "kind": "profile", "mode": "local", "queries": 5, "qlo": 60, "qhi": 700,
         "targets": 60_000, "tlo": 0, "thi": 0, "top_k": 50},
        # A burst of mixed requests at a server: protein searches and read batches.
        {"name": "serving_burst", "kind": "serving", "searches": 9, "qlo": 50, "qhi": 2000, "targets": 50_000,
         "batches": 4, "reads_lo": 500, "reads_hi": 20_000},
        # A small batch of reads from the host, results back on the host.
        {"name": "reads_small", "kind": "reads", "reads": 1000, "len_a": 150, "len_b": 150, "window": 500,
         "on_device": False},
        # A sequencing run's reads in windows of a genome, everything resident.
        {"name": "reads_large", "kind": "reads", "reads": 1_000_000, "len_a": 150, "len_b": 250, "window": 500,
         "on_device": True},
        # Pairwise alignment of assembled DNA: end to end, all pairs of a batch.
        {"name": "long_global", "kind": "long", "mode": "global", "pairs": 64, "lo": 10_000, "hi": 100_000},
        # A few long pairs, best local region.
        {"name": "long_local", "kind": "long", "mode": "local", "pairs": 7, "lo": 10_000, "hi": 60_000},
        # Rescoring of a candidate list: explicit protein pairs, ragged lengths.
        {"name": "pairs_local", "kind": "pairs", "mode": "local", "pairs": 20_000, "lo": 50, "hi": 1500},
        # Distances for clustering or a guide tree: end-to-end protein pairs.
        {"name": "pairs_global", "kind": "pairs", "mode": "global", "pairs": 15_001, "lo": 50, "hi": 1500},
        # Scores of ragged reads for a caller that owns all device memory.
        {"name": "scores_noalloc", "kind": "noalloc", "mode": "semi", "pairs": 30_011, "len_a": 36, "len_b": 301,
         "window": 411},
    ]


def draw(rng):
    def logu(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["search", "search", "profile", "serving", "reads", "reads", "long", "long", "pairs",
                       "pairs", "noalloc"])
    if kind in ("search", "profile"):
        qlo = logu(50, 600)
        queries = logu(1, 32)
        case = {"kind": kind, "mode": rng.choice(["local", "local", "global", "semi"]), "queries": queries,
                "qlo": qlo, "qhi": min(5000, qlo * rng.randint(1, 9)), "targets": logu(2000, 200_000),
                "tlo": 0, "thi": 0, "top_k": rng.choice([1, 10, 10, 50])}
        if rng.random() < 0.3:
            case["tlo"], case["thi"] = 50, rng.randint(300, 700)
        if kind == "search":
            case["host_queries"] = rng.random() < 0.5
        return case
    if kind == "serving":
        return {"kind": kind, "searches": rng.randint(3, 12), "qlo": 50, "qhi": rng.randint(300, 2000),
                "targets": logu(10_000, 60_000), "batches": rng.randint(1, 6), "reads_lo": 500,
                "reads_hi": logu(1000, 30_000)}
    if kind == "reads":
        reads = logu(1000, 700_000)
        len_a = rng.choice([75, 100, 101, 125, 150, 151])
        len_b = rng.choice([len_a, len_a, 250, 251])
        return {"kind": kind, "reads": reads, "len_a": len_a, "len_b": len_b,
                "window": len_b + rng.randint(60, 260), "on_device": reads > 20_000}
    if kind == "long":
        hi = logu(15_000, 100_000)
        return {"kind": kind, "mode": rng.choice(["global", "local"]), "pairs": logu(1, 64), "lo": 10_000, "hi": hi}
    if kind == "pairs":
        lo = logu(30, 120)
        return {"kind": kind, "mode": rng.choice(["local", "global", "semi"]), "pairs": logu(1000, 60_000),
                "lo": lo, "hi": rng.randint(400, 1800)}
    len_a = rng.randint(36, 150)
    return {"kind": kind, "mode": rng.choice(["local", "global", "semi"]), "pairs": logu(1000, 100_000),
            "len_a": len_a, "len_b": len_a + rng.randint(0, 151), "window": rng.randint(310, 600)}


# ---- inputs ----

def _lognormal_lengths(n):
    """Quantiles of the protein databases' length distribution (median 300, sigma 0.7)."""
    p = (torch.arange(n, dtype=torch.float64) + 0.5) / n
    x = torch.exp(math.log(300.0) + 0.7 * torch.special.ndtri(p))
    return x.round().clamp(1, 35_000).long()


def _uniform_lengths(n, lo, hi):
    return (lo + (torch.arange(n, dtype=torch.float64) + 0.5) / n * (hi + 1 - lo)).long()


def _log_lengths(n, lo, hi):
    p = (torch.arange(n, dtype=torch.float64) + 0.5) / n
    return torch.exp(math.log(lo) + p * (math.log(hi) - math.log(lo))).round().long()


def _target_lengths(case):
    if case["thi"]:
        return _uniform_lengths(case["targets"], case["tlo"], case["thi"])
    return _lognormal_lengths(case["targets"])


def _pair_lengths(case):
    """Lengths of the protein pairs' sequences: (queries, targets)."""
    nq = max(1, case["pairs"] // 8)
    return _log_lengths(nq, case["lo"], case["hi"]), _log_lengths(max(1, case["pairs"] // 5), case["lo"], case["hi"])


def _serving_sizes(case):
    return (_log_lengths(case["searches"], case["qlo"], case["qhi"]),
            _log_lengths(case["batches"], case["reads_lo"], case["reads_hi"]))


def _read_lengths(case, n):
    if case["kind"] == "noalloc":
        return _uniform_lengths(n, case["len_a"], case["len_b"])
    return torch.where(torch.arange(n) < n // 2, case["len_a"], case["len_b"]).long()


def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1_000_003 + 170101575)
    return g


def _shuffled(lengths, g):
    return lengths[torch.randperm(len(lengths), generator=g, device="cuda").cpu()]


def _offsets(lengths):
    off = np.zeros(len(lengths) + 1, np.uint64)
    off[1:] = np.cumsum(lengths.numpy())
    return off


def _residues(count, g):
    """Protein residues with the background frequencies of natural proteins."""
    cdf = torch.as_tensor(np.cumsum(workloads.protein_background()), dtype=torch.float32, device="cuda")
    u = torch.rand(count, generator=g, device="cuda")
    return torch.bucketize(u, cdf[:-1].contiguous(), right=True).to(torch.uint8)


def _copies(ref, origins, length, subs, indels, letters, g):
    """[len(origins), length] copies of `ref` from each origin with substitutions and indels."""
    n, shape = len(origins), (len(origins), length)
    event = torch.rand(shape, generator=g, device="cuda")
    extra = torch.rand(shape, generator=g, device="cuda").clamp_min(1e-6).log2().neg().long()   # geometric
    step = torch.where(event < indels / 2, 0, torch.where(event < indels, 2 + extra, 1))
    at = origins[:, None] + torch.cumsum(step, 1)
    at -= step[:, :1]
    got = ref[at.clamp_(max=len(ref) - 1)].long()
    del at, extra
    shift = torch.randint(1, letters, shape, generator=g, device="cuda")
    other = (torch.rand(shape, generator=g, device="cuda") < subs) | (step == 0)
    return torch.where(other, (got + shift) % letters, got).to(torch.uint8)


def _homologs(queries, q_off, targets, t_off, picks, g):
    """Writes a mutated piece of a query into each picked target: the related
    sequences that a search finds.  picks: (query, target) pairs."""
    lens = [int(min(q_off[q + 1] - q_off[q], t_off[t + 1] - t_off[t])) for q, t in picks]
    longest = max(lens)
    origins = torch.tensor([int(q_off[q]) for q, _ in picks], device="cuda")
    pieces = _copies(queries, origins, longest, 0.35, 0.02, 20, g)
    for (q, t), n, piece in zip(picks, lens, pieces):
        targets[int(t_off[t]):int(t_off[t]) + n] = piece[:n]


def _proteins(lengths, g):
    off = _offsets(lengths)
    return _residues(int(off[-1]), g), off


def _reads(lengths, window, g, genome_len=10_000_000):
    """(genome, read codes, read offsets, pairs): reads sampled from a random
    genome (1% substitutions, 0.1% indels), each with a window around it."""
    n = len(lengths)
    genome = torch.randint(0, 4, (genome_len,), generator=g, device="cuda").to(torch.uint8)
    off = _offsets(lengths)
    codes = torch.empty(int(off[-1]), dtype=torch.uint8, device="cuda")
    dev_len = lengths.cuda()
    origins = (torch.rand(n, generator=g, device="cuda", dtype=torch.float64) * (genome_len - 2048)).long()
    for lo in range(0, n, 262_144):
        hi = min(n, lo + 262_144)
        longest = int(lengths[lo:hi].max())
        block = _copies(genome, origins[lo:hi], longest, 0.01, 0.001, 4, g)
        keep = torch.arange(longest, device="cuda")[None, :] < dev_len[lo:hi, None]
        first, last = int(off[lo]), int(off[hi])
        codes[first:last] = block[keep]
    pairs = np.zeros(n, dsa.PAIR_DTYPE)
    pairs["query_id"] = np.arange(n)
    pairs["t_offset"] = (origins + (dev_len - window) // 2).clamp(0, genome_len - window).cpu().numpy()
    pairs["t_len"] = window
    return genome.cpu().numpy(), codes, off, pairs


_context = None


def _ctx():
    """The program's one context."""
    global _context
    if _context is None:
        _context = dsa.Context(0)
    return _context


def prepare(case, seed):
    g = _generator(seed)
    ctx = _ctx()
    kind = case["kind"]
    if kind in ("search", "profile"):
        queries, q_off = _proteins(_shuffled(_log_lengths(case["queries"], case["qlo"], case["qhi"]), g), g)
        targets, t_off = _proteins(_shuffled(_target_lengths(case), g), g)
        where = torch.randperm(case["targets"], generator=g, device="cuda")[:8 * case["queries"]].cpu().tolist()
        _homologs(queries, q_off, targets, t_off, [(k // 8, t) for k, t in enumerate(where)], g)
        s = {"case": case, "ctx": ctx, "db": ctx.load(targets.cpu().numpy(), t_off, 24),
             "matrix": workloads.blosum62()}
        queries = queries.cpu().numpy()
        if kind == "profile":
            s["queries"] = ctx.load(queries, q_off, 24)
            noise = torch.randint(-1, 2, (len(queries), 24), generator=g, device="cuda").cpu().numpy()
            s["pssm"] = (s["matrix"][queries] + noise).astype(np.int8)
        elif case["host_queries"]:
            s["q_codes"], s["q_off"] = queries, q_off
        else:
            s["queries"] = ctx.load(queries, q_off, 24)
        return s
    if kind == "serving":
        q_len, counts = _serving_sizes(case)
        targets, t_off = _proteins(_shuffled(_lognormal_lengths(case["targets"]), g), g)
        counts = counts.tolist()
        genome, codes, off, pairs = _reads(torch.full((sum(counts),), 150), 500, g)
        codes = codes.cpu().numpy()
        requests = []
        for n in _shuffled(q_len, g).tolist():
            requests.append((_residues(n, g).cpu().numpy(), np.array([0, n], np.uint64), None))
        at = 0
        for k, n in enumerate(counts):
            part = pairs[at:at + n].copy()
            part["query_id"] -= at
            read = codes[int(off[at]):int(off[at + n])]
            requests.insert(3 * k + 2, (read, off[at:at + n + 1] - off[at], part))
            at += n
        return {"case": case, "server": dsa.Server(0), "requests": requests,
                "proteins": ctx.load(targets.cpu().numpy(), t_off, 24),
                "genome": ctx.load(genome, np.array([0, len(genome)], np.uint64), 4),
                "blosum": workloads.blosum62(), "dna": workloads.dna_matrix(*READ[:2])}
    if kind == "reads":
        genome, codes, off, pairs = _reads(_shuffled(_read_lengths(case, case["reads"]), g), case["window"], g)
        s = {"case": case, "ctx": ctx, "db": ctx.load(genome, np.array([0, len(genome)], np.uint64), 4),
             "matrix": workloads.dna_matrix(*READ[:2]), "last": None}
        if case["on_device"]:
            s["queries"] = ctx.load(codes.cpu().numpy(), off, 4)
            s["pairs"] = torch.from_numpy(pairs.view(np.uint8)).cuda()
        else:
            s["q_codes"], s["q_off"], s["pairs"] = codes.cpu().numpy(), off, pairs
        return s
    if kind == "long":
        lens = _shuffled(_log_lengths(case["pairs"], case["lo"], case["hi"]), g).tolist()
        first = [torch.randint(0, 4, (n,), generator=g, device="cuda").to(torch.uint8) for n in lens]
        zero = torch.zeros(1, dtype=torch.long, device="cuda")
        second = [_copies(x, zero, len(x), 0.05, 0.01, 4, g)[0] for x in first]
        off = _offsets(torch.tensor(lens))
        pairs = np.zeros(len(lens), dsa.PAIR_DTYPE)
        pairs["query_id"] = pairs["target_id"] = np.arange(len(lens))
        pairs["t_len"] = lens
        return {"case": case, "ctx": ctx, "queries": ctx.load(torch.cat(first).cpu().numpy(), off, 4),
                "db": ctx.load(torch.cat(second).cpu().numpy(), off, 4), "pairs": pairs,
                "matrix": workloads.dna_matrix(*LONG[:2])}
    if kind == "pairs":
        q_len, t_len = _pair_lengths(case)
        q_len, t_len = _shuffled(q_len, g), _shuffled(t_len, g)
        queries, q_off = _proteins(q_len, g)
        targets, t_off = _proteins(t_len, g)
        related = range(0, len(t_len), 2)
        _homologs(queries, q_off, targets, t_off, [(t // 2 % len(q_len), t) for t in related], g)
        k = np.arange(case["pairs"])
        pairs = np.zeros(case["pairs"], dsa.PAIR_DTYPE)
        pairs["target_id"] = k % len(t_len)
        pairs["query_id"] = np.where(pairs["target_id"] % 2 == 0, pairs["target_id"] // 2 % len(q_len),
                                     k * 7 % len(q_len))
        pairs["t_len"] = t_len.numpy()[pairs["target_id"]]
        return {"case": case, "ctx": ctx, "queries": ctx.load(queries.cpu().numpy(), q_off, 24),
                "db": ctx.load(targets.cpu().numpy(), t_off, 24), "pairs": pairs,
                "matrix": workloads.blosum62()}
    n = case["pairs"]
    genome, codes, off, pairs = _reads(_shuffled(_read_lengths(case, n), g), case["window"], g)
    return {"case": case, "q_codes": codes, "q_off": torch.from_numpy(off.view(np.int64)).cuda(),
            "t_codes": torch.from_numpy(genome).cuda(), "t_off": torch.tensor([0, len(genome)], device="cuda"),
            "pairs": torch.from_numpy(pairs.view(np.uint8)).cuda(),
            "matrix": torch.from_numpy(workloads.dna_matrix(*READ[:2])).cuda(),
            "out": torch.empty(3, n, dtype=torch.int32, device="cuda")}


# ---- one pass ----

_FIELDS = [0, 1, 2, 3, 4, 5, 6, 7, 12]   # a hit's 32-bit words but its place in the CIGAR array


def _padded(words, room):
    """CIGAR words at the front of an array of `room` entries (how many there are depends on the residues)."""
    out = np.zeros(room, np.int32)
    out[:len(words)] = words.view(np.int32)
    return out


def _host(res, words_per_hit):
    """Hits and CIGARs (in hit order) of a result, as a program reads them."""
    hits, cigar = res.hits(), res.cigar()
    res.free()
    off, n = hits["cigar_off"].astype(np.int64), hits["cigar_len"].astype(np.int64)
    ends = np.cumsum(n)
    total = int(ends[-1]) if len(ends) else 0
    words = cigar[np.repeat(off - (ends - n), n) + np.arange(total)]
    hits = hits.view(np.int32).reshape(-1, 14)[:, _FIELDS]
    return {"hits": hits, "cigar": _padded(words, words_per_hit * len(hits))} if words_per_hit else {"hits": hits}


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "search":
        ctx, mode = s["ctx"], MODES[case["mode"]]
        if case["host_queries"]:
            res = ctx.align_batch(s["db"], s["q_codes"], s["q_off"], s["matrix"], *PROTEIN, mode=mode,
                                  top_k=case["top_k"])
        else:
            res = ctx.align(s["db"], s["queries"], s["matrix"], *PROTEIN, mode=mode, top_k=case["top_k"])
        ctx.traceback(res)
        return _host(res, 1024)
    if kind == "profile":
        return _host(s["ctx"].align_pssm(s["db"], s["queries"], s["pssm"], *PROTEIN, mode=MODES[case["mode"]],
                                         top_k=case["top_k"]), 0)
    if kind == "serving":
        server = s["server"]
        tickets = []
        for codes, off, pairs in s["requests"]:
            if pairs is None:
                tickets.append(server.submit(s["proteins"], codes, off, s["blosum"], *PROTEIN, top_k=10))
            else:
                tickets.append(server.submit(s["genome"], codes, off, s["dna"], *READ[2:], mode=dsa.SEMIGLOBAL,
                                             free_ends=WINDOW_ENDS, pairs=pairs))
        server.drain()
        return [_host(server.poll(t)[0], 16 if r[2] is not None else 1024) for t, r in zip(tickets, s["requests"])]
    if kind == "reads":
        ctx = s["ctx"]
        if case["on_device"]:
            res = ctx.align(s["db"], s["queries"], s["matrix"], *READ[2:], mode=dsa.SEMIGLOBAL,
                            free_ends=WINDOW_ENDS, pairs=s["pairs"], flags=dsa.RESULTS_ON_DEVICE)
            ctx.traceback(res)
            ctx.sync()
            out = {"hits": res.device_hits().clone().view(torch.int32), "cigar": _padded(res.cigar(), 16 * case["reads"])}
            res.free()
            return out
        res = ctx.align_batch(s["db"], s["q_codes"], s["q_off"], s["matrix"], *READ[2:], mode=dsa.SEMIGLOBAL,
                              free_ends=WINDOW_ENDS, pairs=s["pairs"])
        ctx.traceback(res)
        return _host(res, 16)
    if kind == "long":
        res = s["ctx"].align(s["db"], s["queries"], s["matrix"], *LONG[2:], mode=MODES[case["mode"]],
                             pairs=s["pairs"])
        s["ctx"].traceback(res)
        return _host(res, case["hi"] // 4)
    if kind == "pairs":
        return _host(s["ctx"].align(s["db"], s["queries"], s["matrix"], *PROTEIN, mode=MODES[case["mode"]],
                                    pairs=s["pairs"]), 0)
    out = s["out"]
    rc = dsa.load_library().dsa_score_pairs_noalloc(
        s["q_codes"].data_ptr(), s["q_off"].data_ptr(), case["pairs"], s["t_codes"].data_ptr(),
        s["t_off"].data_ptr(), 1, s["pairs"].data_ptr(), case["pairs"], MODES[case["mode"]], WINDOW_ENDS,
        s["matrix"].data_ptr(), 4, *READ[2:], case["window"], out[0].data_ptr(), out[1].data_ptr(),
        out[2].data_ptr(), torch.cuda.current_stream().cuda_stream)
    if rc != dsa.OK:
        raise dsa.DsaError(rc, "dsa_score_pairs_noalloc")
    return {"score": out[0], "q_end": out[1], "t_end": out[2]}


# ---- what a pass cannot do without ----

def _cells(case):
    """(DP cells, input residues, results) of one pass."""
    kind = case["kind"]
    if kind in ("search", "profile"):
        q = int(_log_lengths(case["queries"], case["qlo"], case["qhi"]).sum())
        t = int(_target_lengths(case).sum())
        return q * t, q + t, case["queries"] * case["top_k"]
    if kind == "serving":
        q_len, counts = _serving_sizes(case)
        q, t, n = int(q_len.sum()), int(_lognormal_lengths(case["targets"]).sum()), int(counts.sum())
        return q * t + n * 150 * 500, q + t + n * 650, case["searches"] * 10 + n
    if kind in ("reads", "noalloc"):
        n = case["reads"] if kind == "reads" else case["pairs"]
        q = int(_read_lengths(case, n).sum())
        return q * case["window"], q + n * case["window"], n
    if kind == "long":
        lens = _log_lengths(case["pairs"], case["lo"], case["hi"])
        return int((lens * lens).sum()), 2 * int(lens.sum()), case["pairs"]
    q_len, t_len = _pair_lengths(case)
    n = case["pairs"]   # half the pairs follow the targets' own query: near the mean product
    return int(n * q_len.double().mean() * t_len.double().mean()), int(q_len.sum() + t_len.sum()), n


def work(case):
    """A DP cell is six operations (two gap states, three maxima, one sum)."""
    cells, residues, results = _cells(case)
    return {"bytes": residues + 56 * results, "flops": 6 * cells}


# ---- the same in 64-bit integers ----

def _gotoh(q, q_len, t, t_len, matrix, o, e, mode, fe):
    """Scores and end cells of padded batches q [n, M], t [n, N]: plain Gotoh, column by column."""
    n, M = q.shape
    N = t.shape[1]
    dev = q.device
    low = -(1 << 40)
    local, semi = mode == dsa.LOCAL, mode == dsa.SEMIGLOBAL
    free = [semi and bool(fe & b) for b in (dsa.FREE_Q_BEGIN, dsa.FREE_Q_END, dsa.FREE_T_BEGIN, dsa.FREE_T_END)]
    i = torch.arange(1, M + 1, device=dev)
    real = i[None, :] <= q_len[:, None]
    edge = -(o + (i - 1) * e)
    H = torch.zeros(n, M + 1, dtype=torch.int64, device=dev)
    if not local and not free[0]:
        H[:, 1:] = edge
    E = torch.full((n, M), low, dtype=torch.int64, device=dev)
    best = torch.zeros(n, dtype=torch.int64, device=dev)
    bi = torch.zeros_like(best)
    bj = torch.zeros_like(best)
    if not local:
        best.fill_(low)
    last = q_len[:, None]
    if free[3]:   # row m from column 0
        best = H.gather(1, last)[:, 0].clone()
        bi = q_len.clone()
    S = matrix.long()
    for j in range(1, N + 1):
        a = t[:, j - 1]
        sub = S[q, a[:, None]]
        top = torch.zeros(n, dtype=torch.int64, device=dev) if local or free[2] else \
            torch.full((n,), -(o + (j - 1) * e), device=dev)
        E = torch.maximum(E - e, H[:, 1:] - o)
        x = torch.maximum(H[:, :-1] + sub, E)
        if local:
            x = x.clamp_min(0)
        # F of row i: the best opening above it; a gap never reopens inside F
        opened = torch.cat([top[:, None], x[:, :-1]], 1) - o + (i - 1) * e
        F = torch.cummax(opened, 1)[0] - (i - 1) * e
        Hn = torch.cat([top[:, None], torch.maximum(x, F)], 1)
        live = j <= t_len
        if local:
            v, r = torch.where(real, Hn[:, 1:], low).max(1)
            r = (Hn[:, 1:] == v[:, None]).long().argmax(1)
            better = live & (v > best)
            best, bi, bj = torch.where(better, v, best), torch.where(better, r + 1, bi), torch.where(better, j, bj)
        else:
            end = j == t_len
            v = Hn.gather(1, last)[:, 0]
            if free[3]:
                better = live & (v > best)
                best, bi, bj = torch.where(better, v, best), torch.where(better, q_len, bi), torch.where(better, j, bj)
            else:
                best, bi, bj = torch.where(end, v, best), torch.where(end, q_len, bi), torch.where(end, j, bj)
            if free[1]:
                col = torch.cat([Hn[:, :1], torch.where(real, Hn[:, 1:], low)], 1)
                v = col.max(1)[0]
                r = (col == v[:, None]).long().argmax(1)
                better = end & ((v > best) | ((v == best) & ((bj > j) | ((bj == j) & (r < bi)))))
                best, bi, bj = torch.where(better, v, best), torch.where(better, r, bi), torch.where(better, j, bj)
        H = torch.where(live[:, None], Hn, H)
    if local:
        bi, bj = torch.where(best > 0, bi, 0), torch.where(best > 0, bj, 0)
    return best, bi - 1, bj - 1


def exact(case, seed):
    """Scores and end cells of the allocation-free call.  The other cases give
    hit records and CIGARs, whole numbers that come from a walk over the
    matrix and have no plain array form."""
    if case["kind"] != "noalloc" or _cells(case)[0] > 2.5e9:
        return None
    s = prepare(case, seed)
    off = s["q_off"]
    q_len = off[1:] - off[:-1]
    pairs = s["pairs"].cpu().numpy().view(dsa.PAIR_DTYPE)
    start = torch.from_numpy(pairs["t_offset"].astype(np.int64)).cuda()
    M, N, n = int(q_len.max()), case["window"], case["pairs"]
    at = (off[:-1, None] + torch.arange(M, device="cuda")).clamp(max=len(s["q_codes"]) - 1)
    q = s["q_codes"][at].long()
    t = s["t_codes"][start[:, None] + torch.arange(N, device="cuda")].long()
    got = _gotoh(q, q_len, t, torch.full((n,), N, device="cuda"), s["matrix"], *READ[2:], MODES[case["mode"]],
                 WINDOW_ENDS)
    return {"score": got[0], "q_end": got[1], "t_end": got[2]}
