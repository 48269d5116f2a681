"""The work that this library is measured on.

Alignment scores, coordinates and paths are whole numbers, so every case is
compared exactly.  Sizes come from the repository's workloads (2 kbp and
200 kbp DNA pairs, 144- to 5,478-residue protein queries against 500,000
subjects, uneven batches up to 20,000 residues, served searches) or lie
between and beyond them.

Kinds of a case:

* align   -- score, end cells and path of one pair (Context.align);
* score   -- score and end cell of one pair (Context.score);
* search  -- one query against a resident database (Database.search);
* batch   -- one run of a plan over many uneven pairs (Batch.run);
* serve   -- requests through the continuous-batching server, all of them
             submitted at once and stepped until the last one is collected.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2211_10769_gb300 import binding
from paper_2211_10769_gb300 import workloads as W

ALGORITHMS = {"local": 0, "global": 1, "semiglobal": 2, "overlap": 3}
OPS_PER_CELL = 10                # Gotoh: E and F three each, H four with the zero floor


def listed():
    return [
        # a protein query realigned against one database hit, the smallest call a search ends in
        dict(name="align_protein_464", kind="align", letters="protein", m=464, n=503, algorithm="local"),
        # two short genes or viral segments
        dict(name="align_dna_2k", kind="align", letters="dna", m=2000, n=2000, algorithm="local"),
        # overlap of two long reads, odd sizes
        dict(name="align_overlap_3k", kind="align", letters="dna", m=3001, n=2753, algorithm="overlap"),
        # resolution only: one virus-sized sequence against a plasmid-sized one, ragged sizes
        dict(name="score_dna_30k", kind="score", letters="dna", m=29903, n=51037, algorithm="local"),
        # end-to-end alignment of two related segments
        dict(name="align_global_100k", kind="align", letters="dna", m=100003, n=99991, algorithm="global"),
        # the long pair of the benchmark
        dict(name="align_dna_200k", kind="align", letters="dna", m=200000, n=200000, algorithm="local"),
        # genome-sized pair
        dict(name="align_dna_1m", kind="align", letters="dna", m=1000000, n=1000000, algorithm="local"),
        # database search with a short, an ordinary and a long query; the short one also takes
        # every subject's score (a statistics pass over the database)
        dict(name="search_144", kind="search", nseq=500000, m=144, k=20, all_scores=True),
        dict(name="search_1000", kind="search", nseq=500000, m=1000, k=20, all_scores=False),
        dict(name="search_5478", kind="search", nseq=500000, m=5478, k=20, all_scores=False),
        # many uneven pairs, DNA and protein in turn, through a plan kept by the program
        dict(name="batch_2000", kind="batch", npairs=2000, shortest=100, longest=20000),
        # an overloaded server: more requests at once than one search
        dict(name="serve_16", kind="serve", nseq=100000, requests=16, longest=5000, k=20, chunks=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["align", "align", "align", "score", "score", "search", "search", "batch", "serve"])
    if kind in ("align", "score"):
        letters = rng.choice(["dna", "dna", "protein"])
        algorithm = rng.choice(["local", "local", "local", "global", "semiglobal", "overlap"])
        top = 35000 if letters == "protein" else (1000000 if algorithm == "local" else 200000)
        m = _log_int(rng, 64, top)
        n = min(top, max(64, int(m * math.exp(rng.uniform(-0.5, 0.5))) | 1))
        return dict(kind=kind, letters=letters, m=m, n=n, algorithm=algorithm)
    if kind == "search":
        nseq = _log_int(rng, 2000, 500000)
        return dict(kind=kind, nseq=nseq, m=_log_int(rng, 50, 5400), k=rng.randint(1, 64),
                    all_scores=rng.random() < 0.3)
    if kind == "batch":
        return dict(kind=kind, npairs=_log_int(rng, 50, 3000), shortest=100, longest=_log_int(rng, 500, 20000))
    return dict(kind=kind, nseq=_log_int(rng, 2000, 100000), requests=rng.randint(2, 16),
                longest=_log_int(rng, 500, 5000), k=20, chunks=4)


# ------------------------------------------------------------------ inputs

def _scoring(letters):
    return W.dna_scoring() if letters == "dna" else W.protein_scoring()


def _random(letters, length, seed):
    return W.uniform_dna(length, seed) if letters == "dna" else W.random_protein(length, seed)


def _pair(case, seed):
    """Two sequences that share a homologous stretch over three quarters of the shorter one."""
    letters, m, n = case["letters"], case["m"], case["n"]
    a = _random(letters, m, 11 * seed + 1)
    span = (3 * min(m, n)) // 4
    at = (m - span) // 2
    core = W.mutate(a[at:at + span], 4 if letters == "dna" else 20, 11 * seed + 2)[:n]
    rest = n - len(core)
    flanks = _random(letters, rest, 11 * seed + 3)
    b = np.concatenate([flanks[:rest // 2], core, flanks[rest // 2:]])
    return a, b


def _database(nseq, queries, seed):
    """Residues and offsets (host arrays) of a protein database: lognormal lengths and background
    composition, two mutated copies of every query among the subjects."""
    lens = W.lognormal_lengths(nseq, 13 * seed + 1)
    g = np.random.default_rng(13 * seed + 2)
    planted = {}
    for k, q in enumerate(queries):
        for c in range(2):
            planted[int(g.integers(0, nseq))] = W.mutate(q, 20, 1000 * seed + 10 * k + c, p_sub=0.15)
    for s, copy in planted.items():
        lens[s] = len(copy)
    offsets = np.zeros(nseq + 1, dtype=np.int64)
    np.cumsum(lens, out=offsets[1:])
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    gen = torch.Generator(device=dev).manual_seed(13 * seed + 3)
    edges = torch.from_numpy(np.cumsum(W.aa_background())[:-1].astype(np.float32)).to(dev)
    res = torch.empty(int(offsets[-1]), dtype=torch.uint8, device=dev)
    step = 1 << 25
    for k in range(0, res.numel(), step):
        u = torch.rand(min(step, res.numel() - k), generator=gen, device=dev)
        res[k:k + step] = torch.bucketize(u, edges, out_int32=True).to(torch.uint8)
    residues = res.cpu().numpy()
    for s, copy in planted.items():
        residues[offsets[s]:offsets[s + 1]] = copy
    return residues, offsets


def _batch_pairs(case, seed):
    """Pairs, every other two related; DNA and protein in turn."""
    g = np.random.default_rng(17 * seed + 1)
    pairs = []
    for k in range(case["npairs"]):
        letters = "dna" if k % 2 == 0 else "protein"
        m = W.log_uniform_int(g, case["shortest"], case["longest"])
        n = W.log_uniform_int(g, case["shortest"], case["longest"])
        if k % 4 < 2:
            a, b = (_random(letters, x, 17 * seed + 10 * k + y) for y, x in enumerate((m, n)))
        else:
            a, b = _pair(dict(letters=letters, m=m, n=n), 17 * seed + k)
        pairs.append((a, b, k % 2))
    return pairs


def _requests(case, seed):
    g = np.random.default_rng(19 * seed + 1)
    return [W.random_protein(W.log_uniform_int(g, 50, case["longest"]), 19 * seed + 2 + k)
            for k in range(case["requests"])]


def prepare(case, seed):
    ctx = binding.Context(0)
    kind = case["kind"]
    st = dict(case=case, ctx=ctx)
    if kind in ("align", "score"):
        a, b = _pair(case, seed)
        st.update(a=torch.from_numpy(a).cuda(), b=torch.from_numpy(b).cuda(), sc=_scoring(case["letters"]))
    elif kind == "search":
        q = W.random_protein(case["m"], 23 * seed + 1)
        residues, offsets = _database(case["nseq"], [q], seed)
        st.update(db=binding.Database(ctx, residues, offsets), q=torch.from_numpy(q).cuda(), sc=W.protein_scoring())
        if case["all_scores"]:
            st["scores"] = torch.empty(case["nseq"], dtype=torch.int32, device="cuda")
    elif kind == "batch":
        scorings = [(s.matrix, s.gap_open, s.gap_extend) for s in (W.dna_scoring(), W.protein_scoring())]
        st["plan"] = binding.Batch(ctx, _batch_pairs(case, seed), scorings,
                                   binding.SW_BATCH_GRAPH | binding.SW_BATCH_AUTOTUNE)
    else:
        queries = _requests(case, seed)
        residues, offsets = _database(case["nseq"], queries[:2], seed)
        st["db"] = binding.Database(ctx, residues, offsets)
        sc = W.protein_scoring()
        st["server"] = binding.Server(ctx, st["db"], sc.matrix, sc.gap_open, sc.gap_extend, mem_budget=8 << 30,
                                      k=case["k"], max_slots=64, chunks=case["chunks"])
        st["queries"] = [torch.from_numpy(q).cuda() for q in queries]
    return st


# --------------------------------------------------------------------- run

def _path(case, cigar):
    """The path's text as bytes, zeros after its end: one length for every path of these sizes."""
    out = np.zeros((case["m"] + case["n"]) // 2 + 64, dtype=np.uint8)
    out[:len(cigar)] = np.frombuffer(cigar, dtype=np.uint8)
    return out


def _hits(hits):
    return np.array(hits, dtype=np.int64).reshape(-1, 2)


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "align":
        sc = st["sc"]
        r = st["ctx"].align(st["a"], st["b"], sc.matrix, sc.gap_open, sc.gap_extend, ALGORITHMS[case["algorithm"]])
        return dict(cells=np.array([r.score, r.a_begin, r.a_end, r.b_begin, r.b_end], dtype=np.int64),
                    cigar=_path(case, r.cigar.encode()))
    if kind == "score":
        sc = st["sc"]
        r = st["ctx"].score(st["a"], st["b"], sc.matrix, sc.gap_open, sc.gap_extend, ALGORITHMS[case["algorithm"]])
        return dict(cells=np.array([r.score, r.a_end, r.b_end], dtype=np.int64))
    if kind == "search":
        sc = st["sc"]
        hits, scores = st["db"].search(st["q"], sc.matrix, sc.gap_open, sc.gap_extend, k=case["k"],
                                       scores_out=st.get("scores"))
        return dict(hits=_hits(hits)) if scores is None else dict(hits=_hits(hits), scores=scores)
    if kind == "batch":
        return dict(cells=np.array([(h.score, h.a_end, h.b_end) for h in st["plan"].run()], dtype=np.int64))
    server = st["server"]
    tickets = [server.submit(q) for q in st["queries"]]
    found = {}
    while len(found) < len(tickets):
        server.step()
        for t in tickets:
            if t not in found:
                hits = server.poll(t)
                if hits is not None:
                    found[t] = _hits(hits)
    return [found[t] for t in tickets]


# -------------------------------------------------------------------- work

def _mean_log_uniform(lo, hi):
    return (hi - lo) / math.log(hi / lo) if hi > lo else float(lo)


def work(case):
    kind = case["kind"]
    if kind in ("align", "score"):
        m, n = case["m"], case["n"]
        return dict(bytes=m + n + 40 + (m // 8 if kind == "align" else 0), flops=OPS_PER_CELL * m * n)
    if kind == "search":
        residues = int(361 * case["nseq"])
        return dict(bytes=residues + case["m"] + (4 * case["nseq"] if case["all_scores"] else 0) + 16 * case["k"],
                    flops=OPS_PER_CELL * residues * case["m"])
    if kind == "batch":
        mean = _mean_log_uniform(case["shortest"], case["longest"])
        return dict(bytes=int(case["npairs"] * (2 * mean + 24)), flops=int(OPS_PER_CELL * case["npairs"] * mean * mean))
    residues = int(361 * case["nseq"])
    mean = _mean_log_uniform(50, case["longest"])
    return dict(bytes=int(residues + case["requests"] * (mean + 16 * case["k"])),
                flops=int(OPS_PER_CELL * residues * case["requests"] * mean))


def tolerance(case):
    return "exact"                      # whole numbers


# ------------------------------------------------------------------- exact

NEG = -(1 << 40)


def _border_top(alg, j, o, e):
    return np.where(j == 0, 0, -(o + (j - 1) * e)) if alg == "global" else np.zeros_like(j)


def _border_left(alg, i, o, e):
    return np.where(i == 0, 0, -(o + (i - 1) * e)) if alg in ("global", "semiglobal") else np.zeros_like(i)


def _align_exact(a, b, mat, o, e, alg):
    """Full matrices, row by row (the gap along a row as a running maximum), and the canonical path."""
    m, n = len(a), len(b)
    mat = mat.astype(np.int64)
    cols = np.arange(n + 1, dtype=np.int64)
    H = np.empty((m + 1, n + 1), np.int64)
    E = np.full((m + 1, n + 1), NEG, np.int64)
    F = np.full((m + 1, n + 1), NEG, np.int64)
    H[0] = _border_top(alg, cols, o, e)
    H[:, 0] = _border_left(alg, np.arange(m + 1, dtype=np.int64), o, e)
    for i in range(1, m + 1):
        F[i, 1:] = np.maximum(F[i - 1, 1:] - e, H[i - 1, 1:] - o)
        x = np.maximum(H[i - 1, :-1] + mat[a[i - 1]][b], F[i, 1:])
        if alg == "local":
            x = np.maximum(x, 0)
        x = np.concatenate([H[i, :1], x])
        E[i, 1:] = np.maximum.accumulate(x + cols * e)[:-1] - o - (cols[1:] - 1) * e
        H[i, 1:] = np.maximum(x[1:], E[i, 1:])
    if alg == "local":
        i, j = (int(v) for v in np.unravel_index(int(np.argmax(H)), H.shape))
    elif alg == "global":
        i, j = m, n
    elif alg == "semiglobal":
        i, j = m, int(np.argmax(H[m]))
    else:
        ends = np.full(H.shape, NEG, np.int64)
        ends[m], ends[:, n] = H[m], H[:, n]
        i, j = (int(v) for v in np.unravel_index(int(np.argmax(ends)), H.shape))
    score, ie, je = int(H[i, j]), i, j
    ops, state = [], "M"
    while i > 0 and j > 0:
        if state == "M":
            if alg == "local" and H[i, j] == 0:
                break
            if H[i, j] == H[i - 1, j - 1] + mat[a[i - 1], b[j - 1]]:
                ops.append("M")
                i, j = i - 1, j - 1
            else:
                state = "I" if H[i, j] == E[i, j] else "D"
        elif state == "I":
            ops.append("I")
            state = "M" if E[i, j] == H[i, j - 1] - o else "I"
            j -= 1
        else:
            ops.append("D")
            state = "M" if F[i, j] == H[i - 1, j] - o else "D"
            i -= 1
    if j == 0 and alg in ("global", "semiglobal"):
        ops += ["D"] * i
        i = 0
    if i == 0 and alg == "global":
        ops += ["I"] * j
        j = 0
    text, k = [], len(ops)
    while k > 0:
        r = k
        while r > 0 and ops[r - 1] == ops[k - 1]:
            r -= 1
        text.append("%d%s" % (k - r, ops[k - 1]))
        k = r
    return (np.array([score, i, ie, j, je], dtype=np.int64) if score or alg != "local" else np.zeros(5, np.int64),
            "".join(text).encode())


def _local_scores(a, b, mat, o, e, dev):
    """Local scores and end cells of a (m) against every row of b (count, n; letters past a
    sequence's end = alphabet size), one anti-diagonal at a time."""
    K = mat.shape[0]
    table = torch.full((K, K + 1), NEG, dtype=torch.int64, device=dev)
    table[:, :K] = torch.from_numpy(mat.astype(np.int64)).to(dev)
    a = a.to(device=dev, dtype=torch.int64)
    b = b.to(device=dev, dtype=torch.int64)
    (m,), (cnt, n) = a.shape, b.shape
    flat = table.reshape(-1)
    arow = a * (K + 1)
    zeros = torch.zeros((cnt, m + 1), dtype=torch.int64, device=dev)
    h1, h2 = zeros.clone(), zeros.clone()          # row i of the last two anti-diagonals (i = 0: the border)
    ee, ff = torch.full_like(zeros, NEG), torch.full_like(zeros, NEG)
    best = torch.zeros((cnt, m), dtype=torch.int64, device=dev)
    bcol = torch.zeros((cnt, m), dtype=torch.int64, device=dev)
    rb = b.flip(1)                                 # column j at n - 1 - j
    for d in range(m + n - 1):                     # cells (i, d - i), 0-based
        lo, hi = max(0, d - n + 1), min(m, d + 1)
        s = flat[arow[lo:hi] + rb[:, n - 1 - d + lo:n - 1 - d + hi]]
        en = torch.maximum(ee[:, lo + 1:hi + 1] - e, h1[:, lo + 1:hi + 1] - o)
        fn = torch.maximum(ff[:, lo:hi] - e, h1[:, lo:hi] - o)
        hn = torch.maximum(torch.maximum(h2[:, lo:hi] + s, en), fn).clamp_(min=0)
        ee[:, lo + 1:hi + 1], ff[:, lo + 1:hi + 1] = en, fn
        h1, h2 = h2, h1
        h1[:, lo + 1:hi + 1] = hn
        if d + 1 < m:
            h1[:, d + 2] = 0                       # the column border of the row that starts next
            h2[:, d + 2] = 0
        better = hn > best[:, lo:hi]
        best[:, lo:hi] = torch.where(better, hn, best[:, lo:hi])
        bcol[:, lo:hi].masked_fill_(better, 0)
        bcol[:, lo:hi] += better * (d + 1 - torch.arange(lo, hi, device=dev))
    score, row = best.max(1)
    row = (best == score[:, None]).to(torch.int8).argmax(1)
    col = bcol.gather(1, row[:, None])[:, 0]
    live = score > 0
    return score, torch.where(live, row + 1, 0), torch.where(live, col, 0)


def exact(case, seed):
    kind = case["kind"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind in ("align", "score"):
        sc = _scoring(case["letters"])
        cells = case["m"] * case["n"]
        if cells <= 2 * 10 ** 7:
            a, b = _pair(case, seed)
            found, cigar = _align_exact(a, b, sc.matrix, sc.gap_open, sc.gap_extend, case["algorithm"])
            return dict(cells=found, cigar=_path(case, cigar)) if kind == "align" else dict(cells=found[[0, 2, 4]])
        if kind == "score" and case["algorithm"] == "local" and case["m"] + case["n"] <= 90000:
            a, b = _pair(case, seed)
            found = _local_scores(torch.from_numpy(a), torch.from_numpy(b)[None], sc.matrix, sc.gap_open,
                                  sc.gap_extend, dev)
            return dict(cells=np.array([int(v[0]) for v in found], dtype=np.int64))
        return None
    if kind == "search" and case["nseq"] * case["m"] <= 8 * 10 ** 7:
        sc = W.protein_scoring()
        q = W.random_protein(case["m"], 23 * seed + 1)
        residues, offsets = _database(case["nseq"], [q], seed)
        lens = np.diff(offsets)
        order = np.argsort(lens, kind="stable")
        res = torch.from_numpy(residues).to(dev)
        scores = np.zeros(case["nseq"], dtype=np.int64)
        for k in range(0, case["nseq"], 20000):
            part = order[k:k + 20000]
            n = int(lens[part].max())
            at = torch.from_numpy(offsets[part]).to(dev)[:, None] + torch.arange(n, device=dev)
            inside = torch.arange(n, device=dev) < torch.from_numpy(lens[part]).to(dev)[:, None]
            b = torch.where(inside, res[at.clamp(max=len(residues) - 1)].to(torch.int64), sc.matrix.shape[0])
            scores[part] = _local_scores(torch.from_numpy(q), b, sc.matrix, sc.gap_open, sc.gap_extend, dev)[0].cpu()
        top = np.lexsort((np.arange(case["nseq"]), -scores))[:case["k"]]
        out = dict(hits=np.stack([top, scores[top]], axis=1).astype(np.int64))
        if case["all_scores"]:
            out["scores"] = scores
        return out
    return None
