"""Performance cases: what a user of this framework has it do, at the sizes it is used at.

Each case is one call, or one chain of calls, through the public entry points
of ``paper_1110_1328_gb300``.  ``listed()`` names the cases that are always
timed, ``draw(rng)`` gives another one of the same ranges, ``prepare`` makes
the inputs on the GPU from a seed, ``run`` is one pass, ``work`` the bytes and
operations a pass cannot do without, and ``exact`` the verification outputs in
64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1110_1328_gb300 as B

DEV = torch.device("cuda", 0)
P31 = (1 << 31) - 1
KEEP_BAYES = (1 << B.ACCEPT) | (1 << B.ACCEPT_AT_MAX)
KEEP_LITE = 1 << B.LITE_ACCEPT


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # the smallest job: all near-duplicates among a few thousand sets, every
        # stage once; what counts is the latency of its launches
        {"name": "search-sets-2k", "op": "search_sets", "n": 2000, "vocab": 10000, "mean": 50, "hashes": 256,
         "rows": 8, "bands": 32, "t": 0.7, "k": 32, "h": 64},
        # signatures of the neighbour lists of a social graph (power-law degrees)
        {"name": "minhash-graph-1m", "op": "minhash", "n": 1000000, "mean": 30, "hashes": 256},
        # signatures of a text corpus over a stored float projection matrix
        {"name": "srp-sparse-20k", "op": "srp_sparse", "n": 20000, "dim": 100000, "mean": 80, "bits": 2048},
        # a batch of new points hashed for a query: the smallest hashing call
        {"name": "srp-dense-1k", "op": "srp_dense", "n": 1000, "d": 384, "bits": 1024, "centers": 100, "margin": 0.0},
        # word-vector sized rows: a width that is no multiple of a tile, an odd count
        {"name": "srp-dense-100k-300", "op": "srp_dense", "n": 99991, "d": 300, "bits": 1024, "centers": 1000,
         "margin": 0.0},
        # a whole collection of embeddings, hashed with the wide margin
        {"name": "srp-dense-1m", "op": "srp_dense", "n": 1000000, "d": 256, "bits": 1024, "centers": 10000,
         "margin": 1e-3},
        # candidates of that collection: many wide bands, heavy overlap between bands
        {"name": "band-dense-1m", "op": "band_dense", "n": 1000000, "d": 256, "centers": 10000, "bits": 1024,
         "rows": 16, "bands": 64},
        # candidates among a graph's neighbour lists: buckets with power-law sizes
        {"name": "band-graph-1m", "op": "band_graph", "n": 1000000, "mean": 30, "hashes": 256, "rows": 3, "bands": 32},
        # Algorithms 1 and 2 over minhash signatures of 32 bits a hash
        {"name": "verify-graph-400k", "op": "verify_graph", "n": 400000, "mean": 30, "hashes": 256, "rows": 3,
         "bands": 32, "t": 0.5, "k": 32, "h": 64},
        # Algorithms 1 and 2 over sign bits, all hashes there from the start
        {"name": "verify-docs-20k", "op": "verify_docs", "n": 20000, "dim": 100000, "mean": 80, "bits": 2048,
         "rows": 8, "bands": 35, "t": 0.7, "k": 32, "h": 128},
        # the other source of candidates, prefix filtering over an inverted index
        {"name": "allpairs-20k", "op": "allpairs", "n": 20000, "dim": 100000, "mean": 80, "t": 0.7},
        # the whole search over a large corpus: two-byte projection, banding,
        # both algorithms over the first 256 hashes, the rest where needed
        {"name": "search-docs-5m", "op": "search_docs", "n": 5000000, "dim": 1 << 22, "bits": 2048, "lazy": 256,
         "rows": 16, "bands": 5, "t": 0.6, "k": 32, "h": 128},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["search_sets", "minhash", "srp_sparse", "srp_dense", "srp_dense", "band_dense", "band_graph",
                     "verify_graph", "verify_docs", "allpairs", "search_docs"])
    if op == "search_sets":
        hashes = rng.choice([128, 256, 512])
        rows, bands = rng.choice([(4, 32), (4, 16), (3, 20)] if hashes == 128 else [(8, 32), (4, 32), (5, 40)])
        return {"op": op, "n": _log_int(rng, 500, 30000), "vocab": _log_int(rng, 5000, 200000),
                "mean": rng.randint(20, 120), "hashes": hashes, "rows": rows, "bands": bands,
                "t": round(rng.uniform(0.5, 0.9), 2), "k": rng.choice([32, 32, 64]), "h": 64}
    if op == "minhash":
        return {"op": op, "n": _log_int(rng, 5000, 1000000), "mean": rng.randint(10, 60),
                "hashes": rng.choice([64, 96, 128, 256, 512])}
    if op == "srp_sparse":
        return {"op": op, "n": _log_int(rng, 1000, 60000), "dim": _log_int(rng, 10000, 150000),
                "mean": rng.randint(30, 160), "bits": rng.choice([128, 256, 384, 512, 1024, 2048])}
    if op == "srp_dense":
        n = _log_int(rng, 200, 1000000)
        d = rng.choice([64, 100, 128, 200, 256, 300, 384, 512, 768])
        bits = rng.choice([128, 256, 512, 1024, 2048])
        if n * d * bits > 2.6e11:
            n = int(2.6e11 / (d * bits))
        return {"op": op, "n": n, "d": d, "bits": bits, "centers": max(10, n // 100),
                "margin": rng.choice([0.0, 0.0, 1e-3])}
    if op == "band_dense":
        n = _log_int(rng, 10000, 1000000)
        return {"op": op, "n": n, "d": rng.choice([64, 128, 256]), "centers": max(20, n // 100), "bits": 1024,
                "rows": 16, "bands": rng.choice([16, 24, 32, 48, 64])}
    if op == "band_graph":
        rows, bands = rng.choice([(3, 32), (3, 21), (4, 32), (4, 50)])
        return {"op": op, "n": _log_int(rng, 20000, 1000000), "mean": rng.randint(15, 40), "hashes": 256,
                "rows": rows, "bands": bands}
    if op == "verify_graph":
        hashes = rng.choice([128, 256, 512])
        return {"op": op, "n": _log_int(rng, 10000, 600000), "mean": rng.randint(15, 40), "hashes": hashes,
                "rows": 3, "bands": 32, "t": round(rng.uniform(0.4, 0.8), 2), "k": rng.choice([32, 32, 64]), "h": 64}
    if op == "verify_docs":
        bits = rng.choice([512, 1024, 2048])
        return {"op": op, "n": _log_int(rng, 2000, 40000), "dim": _log_int(rng, 20000, 120000),
                "mean": rng.randint(40, 120), "bits": bits, "rows": 8, "bands": rng.choice([20, 35, 48]),
                "t": round(rng.uniform(0.5, 0.9), 2), "k": rng.choice([32, 32, 64, 128]), "h": 128}
    if op == "allpairs":
        return {"op": op, "n": _log_int(rng, 2000, 30000), "dim": _log_int(rng, 20000, 150000),
                "mean": rng.randint(30, 100), "t": round(rng.uniform(0.6, 0.9), 2)}
    n = _log_int(rng, 50000, 5000000)
    return {"op": op, "n": n, "dim": 1 << rng.randint(19, 22), "bits": rng.choice([1024, 2048]),
            "lazy": rng.choice([256, 256, 512]), "rows": 16, "bands": rng.randint(3, 5 if n > 3000000 else 9),
            "t": round(rng.uniform(0.55, 0.8), 2), "k": 32, "h": 128}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

class _Draws:
    """Seeded draws on the GPU."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(int(seed) * 7919 + 17)

    def uniform(self, n):
        return torch.rand(n, generator=self.g, device=DEV, dtype=torch.float64)

    def normal(self, *shape):
        return torch.randn(shape, generator=self.g, device=DEV, dtype=torch.float32)

    def integers(self, lo, hi, n):
        return torch.randint(lo, hi, (n,), generator=self.g, device=DEV)

    def permutation(self, n):
        return torch.randperm(n, generator=self.g, device=DEV)


def _lognormal_lengths(r, n, mean, sigma=0.8, least=2):
    z = torch.erfinv(2 * r.uniform(n).clamp(1e-12, 1 - 1e-12) - 1) * math.sqrt(2)
    return torch.exp(math.log(mean) - sigma * sigma / 2 + sigma * z).round().clamp_min(least).to(torch.int64)


def _power_lengths(r, n, lo=5, hi=20000):
    """p(l) ~ l^-2 on [lo, hi]."""
    u = r.uniform(n)
    return (1.0 / (1.0 / lo + u * (1.0 / (hi + 1) - 1.0 / lo))).floor().clamp(lo, hi).to(torch.int64)


def _planted_rows(r, lens, sample, n_groups, dim):
    """Rows of sample()d ids; the first rows are groups of 2..5 members, a base
    and variants that redraw a fraction U[0.1, 0.4] of its draws.  Repeated
    ids within a row merge: (row, id, draws), sorted by row, then id."""
    n = lens.numel()
    sizes = r.integers(2, 6, n_groups)
    base = torch.arange(n, device=DEV)
    end = torch.cumsum(sizes, 0)
    starts, n_grouped = end - sizes, min(n, int(end[-1].item()))
    base[:n_grouped] = torch.repeat_interleave(starts, sizes)[:n_grouped]
    lens = lens[base]
    row = torch.repeat_interleave(torch.arange(n, device=DEV), lens)
    first = torch.cumsum(lens, 0) - lens
    ids = sample(row.numel())
    frac = 0.1 + 0.3 * r.uniform(n)
    head = int(lens[:n_grouped].sum().item())          # the draws of the grouped rows
    rh = row[:head]
    src = first[base[rh]] + (torch.arange(head, device=DEV) - first[rh])
    keep = r.uniform(head) >= frac[rh]
    ids[:head] = torch.where(keep, ids[src], ids[:head])
    key, draws = torch.unique(row * dim + ids, sorted=True, return_counts=True)
    row = key // dim
    return row, key - row * dim, draws


def _indptr(row, n):
    p = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    p[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    return p


def _sets(r, n, vocab, mean):
    """Sets over a vocabulary, a tenth of them seeds of near-duplicate groups."""
    lens = _lognormal_lengths(r, n, mean).clamp_max(vocab // 2)
    row, ids, _ = _planted_rows(r, lens, lambda m: r.integers(0, vocab, m), max(1, n // 20), vocab)
    return _indptr(row, n), ids.to(torch.int32)


def _graph(r, n, mean):
    """Neighbour lists of a Chung-Lu graph with power-law degrees (exponent 2.1)."""
    w = (torch.arange(n, device=DEV, dtype=torch.float64) + 10.0) ** (-1.0 / 1.1)
    cdf = torch.from_numpy(np.cumsum(w.cpu().numpy())).to(DEV)   # on the host: the same sums every time
    cdf = cdf / cdf[-1].item()
    pick = lambda m: torch.searchsorted(cdf, r.uniform(m)).clamp_max(n - 1)
    m = int(n * mean / 2)
    u, v = pick(m), pick(m)
    lone = torch.bincount(torch.cat([u, v])[torch.cat([u != v, u != v])], minlength=n) == 0
    lu = torch.nonzero(lone).ravel()
    lv = pick(lu.numel())
    u, v = torch.cat([u, lu]), torch.cat([v, torch.where(lv == lu, (lv + 1) % n, lv)])
    ok = u != v
    u, v = u[ok], v[ok]
    key = torch.unique(torch.cat([u * n + v, v * n + u]))
    row = key // n
    return _indptr(row, n), (key - row * n).to(torch.int32)


def _docs(r, n, dim, lens, n_groups):
    """tf-idf rows of unit norm over Zipf(1.1) terms."""
    perm = r.permutation(dim)
    top = float(dim) ** -0.1

    def terms(m):
        rank = (1.0 + r.uniform(m) * (top - 1.0)) ** -10.0
        return perm[rank.floor().clamp(1, dim).to(torch.int64) - 1]

    row, ids, draws = _planted_rows(r, lens, terms, n_groups, dim)
    tf = draws.to(torch.float64) + torch.floor(torch.log(r.uniform(row.numel()).clamp_min(1e-300)) / math.log(0.5))
    df = torch.bincount(ids, minlength=dim)
    w = torch.log1p(tf) * torch.log(n / df[ids].clamp_min(1).to(torch.float64)).clamp_min(1e-3)
    sq = torch.zeros(n, dtype=torch.int64, device=DEV)    # in whole numbers: the same sums every time
    sq.index_add_(0, row, (w * w * 2.0 ** 24).round().to(torch.int64))
    w = w / torch.sqrt(sq[row].clamp_min(1).to(torch.float64) * 2.0 ** -24)
    return _indptr(row, n), ids.to(torch.int32), w.to(torch.float32)


def _points(r, n, d, centers):
    """A mixture on the unit sphere, noise norm about 0.15."""
    c = r.normal(centers, d)
    c = c / torch.linalg.vector_norm(c, dim=1, keepdim=True)
    return (c[r.integers(0, centers, n)] + r.normal(n, d) * (0.15 / math.sqrt(d))).contiguous()


def _coeffs(r, n):
    return r.integers(1, P31, n).to(torch.int32), r.integers(0, P31, n).to(torch.int32)


def _zeros(n, dtype):
    return torch.zeros(n, dtype=dtype, device=DEV)


class _State:
    pass


def _capacity(case, count):
    """Room for the candidates: what inputs of this size may have, not the
    count of these; `count` where that is more."""
    n, op = case["n"], case["op"]
    if op in ("band_graph", "verify_graph", "search_sets"):   # the count varies with the hash functions
        return max(count, (64 if op == "search_sets" else 400) * n)
    room = {"band_dense": 1.6, "search_docs": 1.25, "verify_docs": 2.5}[op]
    return max(count, int(room * _pairs_expected(case)) + 20 * n)


def _candidate_buffers(s, sig, kind, rows, bands):
    """Workspace and pair list of the banding call, after a count-only call."""
    s.ws = _zeros(B.blsh_lsh_candidates_workspace(sig.shape[0], kind, rows, bands), torch.uint8)
    s.n_pairs = _zeros(1, torch.int64)
    B.blsh_lsh_candidates(s.ctx, sig, kind, rows, bands, None, s.n_pairs, s.ws)
    B.blsh_status(s.ctx)
    s.pairs = _zeros((_capacity(s.case, int(s.n_pairs.item())), 2), torch.int32)


def _outcome_buffers(s, P, levels):
    s.status, s.lstatus = _zeros(P, torch.uint8), _zeros(P, torch.uint8)
    s.n_used, s.m, s.est = _zeros(P, torch.int16), _zeros(P, torch.int16), _zeros(P, torch.float32)
    s.sim, s.hist = _zeros(P, torch.float64), _zeros(levels, torch.int64)


def _params(case, kind, n_max):
    return B.make_params(kind=kind, t=case["t"], k=case["k"], n_max=n_max, h=case["h"])


def prepare(case, seed):
    s, r, op, n = _State(), _Draws(seed), case["op"], case["n"]
    s.case, s.op = case, op
    s.ctx = B.Context(0)
    B.blsh_ctx_reserve(s.ctx, n)
    if op in ("minhash", "search_sets", "band_graph", "verify_graph"):
        if op == "search_sets":
            s.indptr, s.indices = _sets(r, n, case["vocab"], case["mean"])
        else:
            s.indptr, s.indices = _graph(r, n, case["mean"])
        s.a, s.b = _coeffs(r, case["hashes"])
        s.values = None
        s.sig = _zeros((n, case["hashes"]), torch.int32)
        if op != "minhash":
            B.blsh_minhash(s.ctx, s.indptr, s.indices, case["hashes"], s.a, s.b, s.sig)
            _candidate_buffers(s, s.sig, B.JACCARD, case["rows"], case["bands"])
        kind, n_max = B.JACCARD, case["hashes"]
    elif op in ("srp_sparse", "verify_docs", "allpairs"):
        lens = _lognormal_lengths(r, n, case["mean"]).clamp_max(case["dim"] // 4)
        s.indptr, s.indices, s.values = _docs(r, n, case["dim"], lens, max(1, n // 100))
        if op == "allpairs":
            nnz = s.indices.numel()
            s.n_pairs, n_dups = _zeros(1, torch.int64), _zeros(1, torch.int64)
            ws = _zeros(B.blsh_allpairs_workspace(n, nnz, case["dim"], 0), torch.uint8)
            B.blsh_allpairs_candidates(s.ctx, s.indptr, s.indices, s.values, case["dim"], case["t"], B.COSINE, None,
                                       s.n_pairs, ws, 0, n_dups)
            B.blsh_status(s.ctx)
            s.max_dups = int(n_dups.item())
            s.ws = _zeros(B.blsh_allpairs_workspace(n, nnz, case["dim"], s.max_dups), torch.uint8)
            s.pairs = _zeros((n * (n - 1) // 2, 2), torch.int32)
            return s
        s.R = r.normal(case["dim"], case["bits"])
        s.sig = _zeros((n, case["bits"] // 32), torch.int32)
        if op == "verify_docs":
            B.blsh_srp_sparse(s.ctx, s.indptr, s.indices, s.values, s.R, s.sig)
            del s.R
            _candidate_buffers(s, s.sig, B.COSINE, case["rows"], case["bands"])
        kind, n_max = B.COSINE, case["bits"]
    elif op in ("srp_dense", "band_dense"):
        s.X, s.R = _points(r, n, case["d"], case["centers"]), r.normal(case["d"], case["bits"])
        nbytes = B.blsh_srp_dense_workspace(n, case["d"], case["bits"])
        s.ws = _zeros(nbytes, torch.uint8) if nbytes else None
        s.sig = _zeros((n, case["bits"] // 32), torch.int32)
        if op == "band_dense":
            B.blsh_srp_dense(s.ctx, s.X, s.R, s.sig, workspace=s.ws)
            del s.X, s.R
            _candidate_buffers(s, s.sig, B.COSINE, case["rows"], case["bands"])
        return s
    else:   # search_docs
        s.indptr, s.indices, s.values = _docs(r, n, case["dim"], _power_lengths(r, n), max(1, n // 50))
        s.codes = B.blsh_gaussian_codes(s.ctx, 1000003 * int(seed) + 31, case["dim"], case["bits"])
        s.sig = _zeros((n, case["bits"] // 32), torch.int32)
        s.need = _zeros(n, torch.uint8)
        B.blsh_srp_sparse_q16_cols(s.ctx, s.indptr, s.indices, s.values, s.codes, s.sig, 0, case["lazy"])
        _candidate_buffers(s, s.sig, B.COSINE, case["rows"], case["bands"])
        s.sig.zero_()
        kind, n_max = B.COSINE, case["bits"]
    if op in ("search_sets", "search_docs", "verify_graph", "verify_docs"):
        s.tab = B.blsh_tables_build(s.ctx, _params(case, kind, n_max))
        _outcome_buffers(s, s.pairs.shape[0], s.tab.levels)
    if op in ("search_sets", "search_docs"):
        s.out, s.lout = _zeros(s.pairs.shape[0], torch.int64), _zeros(s.pairs.shape[0], torch.int64)
        s.n_out = _zeros(2, torch.int64)
    if op in ("verify_graph", "verify_docs"):   # the candidates are there before the call
        B.blsh_lsh_candidates(s.ctx, s.sig, kind, case["rows"], case["bands"], s.pairs, s.n_pairs, s.ws)
        B.blsh_status(s.ctx)
        del s.ws
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _verify_both(s):
    B.blsh_verify_both(s.ctx, s.tab, s.pairs, s.sig, s.status, s.n_used, s.m, s.est, s.hist, s.indptr, s.indices,
                       s.values, s.lstatus, s.sim, P_dev=s.n_pairs)


def _band(s, kind):
    B.blsh_lsh_candidates(s.ctx, s.sig, kind, s.case["rows"], s.case["bands"], s.pairs, s.n_pairs, s.ws)


def _compact(s):
    B.blsh_compact(s.ctx, s.status, KEEP_BAYES, s.out, s.n_out[0:1], P_dev=s.n_pairs)
    B.blsh_compact(s.ctx, s.lstatus, KEEP_LITE, s.lout, s.n_out[1:2], P_dev=s.n_pairs)


def _outcomes(s):
    return {"status": s.status, "n_used": s.n_used, "m": s.m, "est": s.est, "hist": s.hist, "lstatus": s.lstatus,
            "sim": s.sim}


def run(s):
    case, op = s.case, s.op
    if op == "minhash":
        B.blsh_minhash(s.ctx, s.indptr, s.indices, case["hashes"], s.a, s.b, s.sig)
        return {"sig": s.sig}
    if op == "srp_sparse":
        B.blsh_srp_sparse(s.ctx, s.indptr, s.indices, s.values, s.R, s.sig)
        return {"sig": s.sig}
    if op == "srp_dense":
        B.blsh_srp_dense(s.ctx, s.X, s.R, s.sig, margin=case["margin"], workspace=s.ws)
        return {"sig": s.sig}
    if op in ("band_dense", "band_graph"):
        _band(s, B.COSINE if op == "band_dense" else B.JACCARD)
        return {"pairs": s.pairs, "n_pairs": s.n_pairs}
    if op == "allpairs":
        B.blsh_allpairs_candidates(s.ctx, s.indptr, s.indices, s.values, case["dim"], case["t"], B.COSINE, s.pairs,
                                   s.n_pairs, s.ws, s.max_dups)
        return {"pairs": s.pairs, "n_pairs": s.n_pairs}
    if op in ("verify_graph", "verify_docs"):
        _verify_both(s)
        return _outcomes(s)
    if op == "search_sets":
        B.blsh_minhash(s.ctx, s.indptr, s.indices, case["hashes"], s.a, s.b, s.sig)
        _band(s, B.JACCARD)
        _verify_both(s)
    else:
        L = case["lazy"]
        B.blsh_srp_sparse_q16_cols(s.ctx, s.indptr, s.indices, s.values, s.codes, s.sig, 0, L)
        _band(s, B.COSINE)
        s.need.zero_()
        B.blsh_verify_both_capped(s.ctx, s.tab, L, s.pairs, s.sig, s.status, s.n_used, s.m, s.est, s.hist, s.indptr,
                                  s.indices, s.values, s.lstatus, s.sim, s.need, P_dev=s.n_pairs)
        B.blsh_srp_sparse_q16_cols(s.ctx, s.indptr, s.indices, s.values, s.codes, s.sig, L, case["bits"] - L,
                                   row_mask=s.need)
        B.blsh_verify_resume(s.ctx, s.tab, s.pairs, s.sig, s.status, s.n_used, s.m, s.est, s.hist, P_dev=s.n_pairs)
    _compact(s)
    return {"sig": s.sig, "pairs": s.pairs, "n_pairs": s.n_pairs, "out": s.out, "lout": s.lout, "n_out": s.n_out,
            **_outcomes(s)}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _pairs_expected(case):
    """About how many candidates the inputs of a case have."""
    n, op = case["n"], case["op"]
    if op == "search_sets":
        return n / 20 * 4
    if op in ("band_graph", "verify_graph"):
        return 100.0 * n                       # 1.0e8 of 1e6 nodes at 3 x 32, mean degree 30
    if op == "band_dense":
        return n * n / (2.0 * case["centers"]) + n * n / 2.0 * case["bands"] * 2.0 ** -case["rows"]
    if op == "search_docs":
        return n * n / 2.0 * case["bands"] * 2.0 ** -case["rows"]
    return n * n / 2.0 * (1.0 - (1.0 - 2.0 ** -8) ** case.get("bands", 35))


def work(case):
    """Each input read once, each output written once.  Operations: two for a
    product and its sum, or for a hash of an element (multiply-add, minimum)."""
    n, op = case["n"], case["op"]
    if op in ("search_docs",):
        nnz, nz = n * 29.0, 8                  # distinct terms of a row: about 29 of its 41 draws
    else:
        nnz, nz = n * float(case.get("mean", 0)), 4 if op in ("minhash", "search_sets", "band_graph",
                                                              "verify_graph") else 8
    rows = nnz * nz + 8 * n
    if op == "minhash":
        return {"bytes": rows + 4.0 * n * case["hashes"], "flops": 2.0 * nnz * case["hashes"]}
    if op == "srp_sparse":
        return {"bytes": rows + 4.0 * min(case["dim"], nnz) * case["bits"] + n * case["bits"] / 8.0,
                "flops": 2.0 * nnz * case["bits"]}
    if op == "srp_dense":
        return {"bytes": 4.0 * (n + case["bits"]) * case["d"] + n * case["bits"] / 8.0,
                "flops": 2.0 * n * case["d"] * case["bits"]}
    P = _pairs_expected(case)
    if op == "band_dense":
        return {"bytes": n * case["rows"] * case["bands"] / 8.0 + 8.0 * P, "flops": 0.0}
    if op == "band_graph":
        return {"bytes": 4.0 * n * min(case["hashes"], case["rows"] * case["bands"]) + 8.0 * P, "flops": 0.0}
    if op == "allpairs":
        return {"bytes": rows + 8.0 * P, "flops": 0.0}
    if op == "verify_graph":                   # the pair, its outcome, the rows its chunks read (once each)
        return {"bytes": 4.0 * n * case["hashes"] + P * (8 + 6) + rows, "flops": 0.0}
    if op == "verify_docs":
        return {"bytes": n * case["bits"] / 8.0 + P * (8 + 6) + rows, "flops": 0.0}
    if op == "search_sets":
        return {"bytes": rows + 4.0 * n * case["hashes"] + P * (8 + 6 + 12), "flops": 2.0 * nnz * case["hashes"]}
    return {"bytes": rows + 2.0 * case["dim"] * case["lazy"] + n * case["lazy"] / 8.0 + P * (8 + 6),
            "flops": 2.0 * nnz * case["lazy"]}


# ---------------------------------------------------------------------------
# the verification outputs in 64 bits
# ---------------------------------------------------------------------------

def _log_binomial_cdf(n, p):
    """log P(Bin(n, p) <= m), m = 0 .. n."""
    m = np.arange(n + 1, dtype=np.float64)
    if p <= 0.0:
        return np.zeros(n + 1)
    if p >= 1.0:
        return np.where(m < n, -np.inf, 0.0)
    lg = np.concatenate([[0.0], np.cumsum(np.log(np.arange(1, n + 1, dtype=np.float64)))])
    return np.logaddexp.accumulate(lg[n] - lg - lg[::-1] + m * math.log(p) + (n - m) * math.log1p(-p))


def _levels(case, kind, n_max):
    """minMatches, [concentrated] and the estimates after each chunk: uniform
    prior, so Pr[X >= x | m of n] = P(Bin(n + 1, x) <= m) over X = S (Jaccard)
    or, divided by the same at 0.5, over X = r = 1 - acos(S) / pi."""
    k, t, eps, delta, gamma = case["k"], case["t"], 0.03, 0.05, 0.03
    to_r = (lambda s: s) if kind == B.JACCARD else (lambda s: 1.0 - math.acos(s) / math.pi)
    out = []
    for n in range(k, n_max + 1, k):
        m = np.arange(n + 1)
        if kind == B.JACCARD:
            est = m / n
            tail = lambda x: _log_binomial_cdf(n + 1, x)[: n + 1]
        else:
            est = np.cos(math.pi * (1.0 - np.maximum(m / n, 0.5)))
            half = _log_binomial_cdf(n + 1, 0.5)[: n + 1]
            tail = lambda x: _log_binomial_cdf(n + 1, x)[: n + 1] - half
        keep = np.exp(tail(to_r(t))) >= eps
        least = int(np.argmax(keep)) if keep.any() else n + 1
        conc = np.zeros(n + 1, bool)
        for i in range(least, n + 1):
            lo, hi = est[i] - delta, min(1.0, est[i] + delta)
            lo = max(0.0, lo) if kind == B.JACCARD else max(0.5, to_r(max(-1.0, lo)))
            conc[i] = math.exp(_tail_at(n, i, lo, kind)) - math.exp(_tail_at(n, i, to_r(hi), kind)) >= 1.0 - gamma
        out.append((least, conc, est))
    return out


def _tail_at(n, m, x, kind):
    """log Pr[X >= x | m of n], one m."""
    def cdf(p):
        if p <= 0.0:
            return 0.0
        if p >= 1.0:
            return -math.inf
        j = np.arange(m + 1, dtype=np.float64)
        terms = _LG[n + 1] - _LG[: m + 1] - _LG[n + 1 - np.arange(m + 1)] + j * math.log(p) + (n + 1 - j) * math.log1p(-p)
        top = terms.max()
        return float(top + math.log(np.exp(terms - top).sum()))
    return cdf(x) if kind == B.JACCARD else cdf(x) - cdf(0.5)


_LG = np.concatenate([[0.0], np.cumsum(np.log(np.arange(1, 4200, dtype=np.float64)))])


def _popcount(v):
    v = v - ((v >> 1) & 0x55555555)
    v = (v & 0x33333333) + ((v >> 2) & 0x33333333)
    v = (v + (v >> 4)) & 0x0F0F0F0F
    return (v * 0x01010101 & 0xFFFFFFFF) >> 24


def _agreements(sig, x, y, level, k, kind):
    """Agreeing hashes of the pairs (x, y) in chunk `level`, in slices."""
    got = torch.empty(x.numel(), dtype=torch.int64, device=DEV)
    step = 1 << 21
    for i in range(0, x.numel(), step):
        if kind == B.JACCARD:
            c = slice(level * k, (level + 1) * k)
            a, b = sig[x[i:i + step], c], sig[y[i:i + step], c]
            got[i:i + step] = (a == b).sum(1)
        else:
            c = slice(level * k // 32, (level + 1) * k // 32)
            d = (sig[x[i:i + step], c] ^ sig[y[i:i + step], c]).to(torch.int64) & 0xFFFFFFFF
            got[i:i + step] = k - _popcount(d).sum(1)
    return got


def _similarities(s, x, y):
    """Exact similarities of the pairs (x, y) from their rows."""
    n = s.case["n"]
    lens = s.indptr[1:] - s.indptr[:-1]
    dim = int(s.indices.max().item()) + 1
    idx = s.indices.to(torch.int64)
    row = torch.repeat_interleave(torch.arange(n, device=DEV), lens)
    key = row * dim + idx
    swap = lens[x] > lens[y]
    x, y = torch.where(swap, y, x), torch.where(swap, x, y)      # x is the shorter row
    if s.values is not None:
        v = s.values.to(torch.float64)
        sq = torch.zeros(n, dtype=torch.float64, device=DEV).index_add_(0, row, v * v)
    got = torch.zeros(x.numel(), dtype=torch.float64, device=DEV)
    ends = torch.cumsum(lens[x], 0)
    at, P = 0, x.numel()
    while at < P:                              # about 1e8 looked-up elements a slice
        before = int(ends[at - 1].item()) if at else 0
        to = max(at + 1, int(torch.searchsorted(ends, torch.tensor([before + 10 ** 8], device=DEV)).item()))
        xs, ys, ls = x[at:to], y[at:to], lens[x[at:to]]
        pair = torch.repeat_interleave(torch.arange(to - at, device=DEV), ls)
        pos = s.indptr[xs][pair] + torch.arange(pair.numel(), device=DEV) - (torch.cumsum(ls, 0) - ls)[pair]
        want = ys[pair] * dim + idx[pos]
        found = torch.searchsorted(key, want).clamp_max(key.numel() - 1)
        hit = key[found] == want
        acc = torch.zeros(to - at, dtype=torch.float64, device=DEV)
        acc.index_add_(0, pair, hit.to(torch.float64) if s.values is None else torch.where(hit, v[pos] * v[found], 0.0))
        got[at:to] = acc / (lens[xs] + lens[ys] - acc) if s.values is None else acc / torch.sqrt(sq[xs] * sq[ys])
        at = to
    return got


def exact(case, seed):
    """Estimates and similarities of the verification calls, from the pairs and
    signatures in hand; the other outputs are whole numbers.  The whole
    searches have none here: their pairs stand in an order of the framework's
    own choice, and 5e6 rows would take minutes."""
    if case["op"] not in ("verify_graph", "verify_docs"):
        return None
    s = prepare(case, seed)
    kind = B.JACCARD if case["op"] == "verify_graph" else B.COSINE
    n_max = case["hashes"] if kind == B.JACCARD else case["bits"]
    P, k = s.pairs.shape[0], case["k"]
    count = int(s.n_pairs.item())
    pairs = s.pairs[:count].to(torch.int64)
    h = min(n_max, -(-case["h"] // k) * k)
    est = torch.zeros(P, dtype=torch.float64, device=DEV)
    open_ = torch.arange(count, device=DEV)             # pairs Algorithm 1 goes on with
    lite = open_                                        # pairs Algorithm 2 has not pruned
    m = torch.zeros(P, dtype=torch.int64, device=DEV)
    for j, (least, conc, value) in enumerate(_levels(case, kind, n_max)):
        if (j + 1) * k <= h:                            # the survivors of both go through the first h hashes
            both = torch.zeros(P, dtype=torch.bool, device=DEV)
            both[open_] = True
            both[lite] = True
            at = torch.nonzero(both).ravel()
        else:
            at = open_
        if not at.numel():
            break
        m[at] += _agreements(s.sig, pairs[at, 0], pairs[at, 1], j, k, kind)
        if (j + 1) * k <= h:
            lite = lite[m[lite] >= least]
        open_ = open_[m[open_] >= least]
        done = torch.from_numpy(conc).to(DEV)[m[open_]]
        if (j + 1) * k == n_max:
            done = torch.ones_like(done)
        est[open_[done]] = torch.from_numpy(value).to(DEV)[m[open_[done]]]
        open_ = open_[~done]
    sim = torch.zeros(P, dtype=torch.float64, device=DEV)
    sim[lite] = _similarities(s, pairs[lite, 0], pairs[lite, 1])
    return {"status": None, "n_used": None, "m": None, "est": est, "hist": None, "lstatus": None, "sim": sim}
