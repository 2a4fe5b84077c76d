"""Performance cases: the calls that programs built on this library make.

Every case goes through the public entry points of ``swgb``: a search through
a plan that the program keeps, the one-shot search of a script, the queued
search of the serving loop, alignments of the best hits, and the search that
allocates nothing.  Lengths, databases and gap penalties are those of the
repository's workloads (``synth``): protein queries of 144-5,478 residues,
lognormal databases (mean 360) up to Swiss-Prot's 570,000 subjects, and
subjects of 5,000-35,000 residues.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2309_09609_gb300 import swgb, synth

#: no drawn search has more cells than the largest listed one
MAX_CELLS = 3.6e12
#: above this many cells a plain 64-bit evaluation takes too long
EXACT_CELLS = 5e10
PAIR_MAX = 4096     # longest subject of the search that allocates nothing


def _search(name, api, queries, query_len, subjects, lengths="lognormal", gap_open=10,
            gap_extend=2, matrix="blosum62", planted=0):
    """A search of `queries` queries (lengths: "paper" log-spaced 144-5478,
    "mixed" lognormal of mean 400, "uniform" 50-2000, "long" 5000-35000, or a
    number) against `subjects` subjects ("lognormal", "uniform" 50-1000 or
    "long" 5000-35000)."""
    return {"name": name, "kind": "search", "api": api, "queries": queries,
            "query_len": query_len, "subjects": subjects, "lengths": lengths,
            "gap_open": gap_open, "gap_extend": gap_extend, "matrix": matrix, "planted": planted}


def _align(name, queries, hits, subjects):
    return {"name": name, "kind": "align", "queries": queries, "query_len": "mixed", "hits": hits,
            "subjects": subjects, "lengths": "lognormal", "gap_open": 10, "gap_extend": 2,
            "matrix": "blosum62", "planted": max(1, queries * hits // 4)}


def listed():
    return [
        # a script scores a few proteins against a small set, arrays in and out
        _search("script-small-set", "oneshot", 3, "mixed", 300),
        # the repository's smallest workload: one 144-residue query, 2,000 subjects
        _search("one-query-2k", "plan", 1, 144, 2000, "uniform"),
        # one average query against a proteome, scores back on the host
        _search("one-query-proteome", "oneshot", 1, 375, 20_000),
        # the serving loop on an idle server: a single request, Swiss-Prot size
        _search("serve-one-request", "async", 1, 375, 570_000, planted=57),
        # the serving loop under load: a batch of requests of mixed lengths
        _search("serve-batch", "async", 5, "mixed", 570_000, planted=57),
        # the paper's query set against a mid-sized database
        _search("paper-queries", "plan", 20, "paper", 100_000, planted=10),
        # a batch job: many uneven queries in one call
        _search("batched-uneven", "plan", 96, "uniform", 100_000, planted=10),
        # long against long, with homologs whose 16-bit scores saturate
        _search("long-sequences", "plan", 4, "long", 500, "long", planted=2),
        # a user's own matrix and gap penalties
        _search("own-matrix", "plan", 7, "mixed", 40_000, gap_open=6, gap_extend=3,
                matrix="own", planted=4),
        # the alignment behind each query's best hit
        _align("align-best-hits", 20, 1, 20_000),
        # the alignments of a result page: 25 hits of each query
        _align("align-result-page", 20, 25, 20_000),
        # a host framework that owns all device memory
        {"name": "caller-memory", "kind": "pairs", "queries": 16, "query_len": "mixed",
         "subjects": 2000, "lengths": "lognormal", "gap_open": 10, "gap_extend": 2,
         "matrix": "blosum62", "planted": 0},
    ]


def _mean_len(spec):
    return {"paper": 1537.0, "mixed": 400.0, "uniform": 1025.0, "long": 20_000.0,
            "lognormal": 360.0}.get(spec, spec)


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges (rng: random.Random), without a name."""
    kind = rng.choice(["search"] * 8 + ["align"] * 2 + ["pairs"])
    if kind == "align":
        queries = _logint(rng, 1, 32)
        c = _align("", queries, _logint(rng, 1, 25), _logint(rng, 1000, 40_000))
    elif kind == "pairs":
        c = {"kind": "pairs", "queries": _logint(rng, 1, 24), "query_len": "mixed",
             "subjects": _logint(rng, 100, 4000), "lengths": "lognormal", "gap_open": 10,
             "gap_extend": 2, "matrix": "blosum62", "planted": 0}
    else:
        api = rng.choice(["oneshot", "plan", "plan", "async"])
        if rng.random() < 0.15:
            c = _search("", api, rng.randint(1, 6), "long", _logint(rng, 50, 700), "long",
                        planted=rng.randint(0, 2))
        else:
            own = rng.random() < 0.2
            go, ge = rng.choice([(6, 3), (9, 2), (12, 1)]) if own else \
                rng.choice([(10, 2), (10, 2), (11, 1)])
            subjects = _logint(rng, 300, 570_000)
            spec = rng.choice(["mixed", "mixed", "uniform", "paper", _logint(rng, 30, 5000)])
            c = _search("", api, _logint(rng, 1, 96), spec, subjects,
                        rng.choice(["lognormal", "lognormal", "uniform"]), go, ge,
                        "own" if own else "blosum62", planted=subjects // 10_000)
        while c["queries"] > 1 and _cells(c) > MAX_CELLS:
            c["queries"] -= 1
    c.pop("name", None)
    return c


def _cells(case):
    db = {"uniform": 525.0}.get(case["lengths"], _mean_len(case["lengths"]))
    if case["kind"] == "align":
        return case["queries"] * case["hits"] * _mean_len(case["query_len"]) * db
    return case["queries"] * _mean_len(case["query_len"]) * case["subjects"] * db


def work(case):
    """Bytes: each residue read once, each score (or alignment record and
    transcript byte) written once.  Operations: the 11 integer additions and
    maxima of a cell of Eq. 1-3."""
    db = {"uniform": 525.0}.get(case["lengths"], _mean_len(case["lengths"]))
    q = case["queries"] * _mean_len(case["query_len"])
    if case["kind"] == "align":
        pairs = case["queries"] * case["hits"]
        return {"bytes": q + pairs * (db + 32 + _mean_len(case["query_len"])),
                "flops": 11.0 * _cells(case)}
    return {"bytes": q + case["subjects"] * db + 4.0 * case["queries"] * case["subjects"],
            "flops": 11.0 * _cells(case)}


# ---- inputs -------------------------------------------------------------------
def _inputs(case, seed):
    """(queries, database, matrix or None) of a case, from the seed alone."""
    rng = np.random.default_rng(seed)
    n, spec = case["queries"], case["query_len"]
    if spec == "paper":
        lens = synth.paper_query_lengths(n)
    elif spec == "mixed":
        sigma = synth.DB_SIGMA
        lens = synth.lognormal_lengths(rng, n, math.log(400.0) - sigma * sigma / 2, sigma, 30, 5000)
    elif spec == "uniform":
        lens = synth.uniform_lengths(rng, n, 50, 2000)
    elif spec == "long":
        lens = synth.uniform_lengths(rng, n, 5000, 35_000)
    else:
        lens = np.full(n, int(spec), dtype=np.int32)
    # the work of a case is fixed by its sizes, not by the luck of the draw
    lens = np.maximum(np.rint(lens * (n * _mean_len(spec) / lens.sum())), 1).astype(np.int32)
    q = synth.random_seqset(rng, lens)
    if case["lengths"] == "uniform":
        dl = synth.uniform_lengths(rng, case["subjects"], 50, 1000)
    elif case["lengths"] == "long":
        dl = synth.uniform_lengths(rng, case["subjects"], 5000, 35_000)
    else:
        dl = synth.lognormal_lengths(rng, case["subjects"],
                                     hi=PAIR_MAX if case["kind"] == "pairs" else 35_000)
    db = synth.random_seqset(rng, dl)
    if case["planted"]:
        long = case["lengths"] == "long"
        synth.plant_homologs(rng, db, q, case["planted"], *((0.05, 0.10) if long else (0.10, 0.20)),
                             prefer_long=long)
    matrix = None
    if case["matrix"] == "own":   # symmetric, mostly negative off the diagonal
        m = rng.integers(-5, 2, size=(24, 24))
        m = np.tril(m) + np.tril(m, -1).T
        np.fill_diagonal(m, rng.integers(4, 13, size=24))
        matrix = m.astype(np.int8)
    return q, db, matrix


def prepare(case, seed):
    """The resident database, the plan a program keeps, and the call's inputs."""
    q, subjects, matrix = _inputs(case, seed)
    state = {"case": case, "q": q, "matrix": matrix}
    dev = torch.device("cuda", 0)
    if case["kind"] == "pairs":
        def to(a):
            return torch.from_numpy(np.ascontiguousarray(a)).to(dev)
        state["args"] = [to(q.res), to(q.offs), to(q.lens),
                         to(subjects.res), to(subjects.offs), to(subjects.lens),
                         torch.empty((len(q), len(subjects)), dtype=torch.int32, device=dev)]
        return state
    db = state["db"] = swgb.Database.from_seqset(subjects, device=0)
    if case["kind"] == "align":   # the pairs a program aligns: each query's best hits
        scores = db.search(q.res, q.lens, case["gap_open"], case["gap_extend"], matrix)
        idx, _ = swgb.top_hits(scores, case["hits"])
        state["pair_query"] = np.repeat(np.arange(len(q), dtype=np.int32), idx.shape[1])
        state["pair_subject"] = np.ascontiguousarray(idx.ravel())
    elif case["api"] != "oneshot":
        state["plan"] = db.plan(len(q), q.total)
        state["out"] = torch.empty((len(q), db.n), dtype=torch.int32, device=dev)
    return state


def run(state):
    """One pass: the scores of every pair, or the alignments of every hit."""
    case, q, matrix = state["case"], state["q"], state["matrix"]
    gaps = (case["gap_open"], case["gap_extend"])
    if case["kind"] == "pairs":
        return swgb.search_pairs_noalloc(*state["args"], *gaps, matrix)
    if case["kind"] == "align":
        found = state["db"].align(q.res, q.lens, state["pair_query"], state["pair_subject"], *gaps,
                                  matrix)
        out = {k: np.array([a[k] for a in found], dtype=np.int32)
               for k in ("score", "q_begin", "q_end", "s_begin", "s_end")}
        # the transcripts, back to back (shorter than 1,024 columns on average)
        ops = np.frombuffer("".join(a["ops"] for a in found).encode(), dtype=np.uint8)
        out["ops"] = np.zeros(1024 * len(found), dtype=np.uint8)
        out["ops"][:ops.size] = ops
        return out
    if case["api"] == "oneshot":
        return state["db"].search(q.res, q.lens, *gaps, matrix)
    if case["api"] == "plan":
        return state["plan"].search(q.res, q.lens, *gaps, matrix, out=state["out"])
    state["plan"].search_async(q.res, q.lens, state["out"], *gaps, matrix)
    state["plan"].wait()
    return state["out"]


# ---- the same scores in 64-bit integers -----------------------------------------
def _exact_scores(query, db, matrix, gap_open, gap_extend, dev):
    """One query against every subject, by antidiagonals, in int64."""
    go, ge, m = gap_open + gap_extend, gap_extend, int(query.size)
    n = len(db)
    out = np.zeros(n, dtype=np.int64)
    sm = torch.full((25, 25), -1000, dtype=torch.int64, device=dev)   # code 24: off the end
    sm[:24, :24] = torch.from_numpy(matrix.astype(np.int64)).to(dev)
    sm = sm.reshape(-1)
    rows = torch.from_numpy(query.astype(np.int64)).to(dev) * 25
    order = np.argsort(db.lens, kind="stable")
    step = max(1, int(2e7 // max(m, 1)))
    for lo in range(0, n, step):
        idx = order[lo:lo + step]
        longest = int(db.lens[idx].max(initial=0))
        if m == 0 or longest == 0:
            continue
        # each subject reversed, so that antidiagonal d is the slice [:, L + m - 1 - d:]
        width = longest + 2 * m
        rev = np.full((idx.size, width), 24, dtype=np.uint8)
        for k, s in enumerate(idx):
            seq = db.seq(int(s))
            rev[k, width - m - seq.size:width - m] = seq[::-1]
        rev = torch.from_numpy(rev).to(dev)
        zero = torch.zeros((idx.size, m + 1), dtype=torch.int64, device=dev)
        h1, h2 = zero.clone(), zero.clone()       # H one and two antidiagonals back, rows 0..m
        e, f = zero - go, zero - go               # E(i, next column), F(next row, j)
        best = torch.zeros(idx.size, dtype=torch.int64, device=dev)
        for d in range(longest + m - 1):
            codes = rev[:, width - m - 1 - d:width - 1 - d].to(torch.int64)
            h = h2[:, :-1] + sm[codes + rows]
            h = torch.maximum(torch.maximum(h, e[:, 1:]), f[:, :-1]).clamp_(min=0)
            best = torch.maximum(best, h.amax(dim=1))
            e[:, 1:] = torch.maximum(e[:, 1:] - ge, h - go)
            f_next = f.clone()
            f_next[:, 1:] = torch.maximum(f[:, :-1] - ge, h - go)
            f = f_next
            h2 = h1
            h1 = zero.clone()
            h1[:, 1:] = h
        out[idx] = best.cpu().numpy()
    return out


def exact(case, seed):
    """The scores in plain 64-bit integers; None where that takes too long,
    and in the place of what is not a score."""
    q, db, matrix = _inputs(case, seed)
    cells = q.total * db.total
    if case["kind"] == "align" or cells > EXACT_CELLS:
        return None
    m = swgb.default_matrix() if matrix is None else matrix
    dev = torch.device("cuda", 0)
    scores = np.stack([_exact_scores(q.seq(i), db, m, case["gap_open"], case["gap_extend"], dev)
                       for i in range(len(q))])
    if case["kind"] == "search" and case["api"] == "oneshot":
        return scores
    return torch.from_numpy(scores)
