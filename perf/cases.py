"""Workloads of the library's public entry points, over the sizes it is used at:
protein searches from one short query against a few thousand proteins up to
twenty queries against 200,000, long DNA pairs, and tracebacks of hits.

``listed()`` names the workloads, ``draw(rng)`` gives others of the same
ranges.  ``prepare`` makes what a program holds before the call (a resident
database, query arrays, a prepared batch), ``run`` is one pass through the
Python front-end, ``work`` the traffic and operations a pass cannot do
without, ``exact`` the scores from a plain 64-bit dynamic program.

Inputs are synthetic: log-normal protein lengths with residues from the
Robinson & Robinson (1991) background law, planted homologs with 10 %
substitutions and 1 % indel events, uniform random DNA with a diverged copy.
Lengths depend on the case alone, residues on the seed.
"""

import math

import numpy as np
import torch

from paper_2412_08308_gb300 import api as sw

# BLOSUM62 (Henikoff & Henikoff 1992) over ARNDCQEGHILKMFPSTWYV, and the
# background composition (Robinson & Robinson 1991) in the same order.
BLOSUM62 = np.array([[int(v) for v in row.split()] for row in """
 4 -1 -2 -2  0 -1 -1  0 -2 -1 -1 -1 -1 -2 -1  1  0 -3 -2  0
-1  5  0 -2 -3  1  0 -2  0 -3 -2  2 -1 -3 -2 -1 -1 -3 -2 -3
-2  0  6  1 -3  0  0  0  1 -3 -3  0 -2 -3 -2  1  0 -4 -2 -3
-2 -2  1  6 -3  0  2 -1 -1 -3 -4 -1 -3 -3 -1  0 -1 -4 -3 -3
 0 -3 -3 -3  9 -3 -4 -3 -3 -1 -1 -3 -1 -2 -3 -1 -1 -2 -2 -1
-1  1  0  0 -3  5  2 -2  0 -3 -2  1  0 -3 -1  0 -1 -2 -1 -2
-1  0  0  2 -4  2  5 -2  0 -3 -3  1 -2 -3 -1  0 -1 -3 -2 -2
 0 -2  0 -1 -3 -2 -2  6 -2 -4 -4 -2 -3 -3 -2  0 -2 -2 -3 -3
-2  0  1 -1 -3  0  0 -2  8 -3 -3 -1 -2 -1 -2 -1 -2 -2  2 -3
-1 -3 -3 -3 -1 -3 -3 -4 -3  4  2 -3  1  0 -3 -2 -1 -3 -1  3
-1 -2 -3 -4 -1 -2 -3 -4 -3  2  4 -2  2  0 -3 -2 -1 -2 -1  1
-1  2  0 -1 -3  1  1 -2 -1 -3 -2  5 -1 -3 -1  0 -1 -3 -2 -2
-1 -1 -2 -3 -1  0 -2 -3 -2  1  2 -1  5  0 -2 -1 -1 -1 -1  1
-2 -3 -3 -3 -2 -3 -3 -3 -1  0  0 -3  0  6 -4 -2 -2  1  3 -1
-1 -2 -2 -1 -3 -1 -1 -2 -2 -3 -3 -1 -2 -4  7 -1 -1 -4 -3 -2
 1 -1  1  0 -1  0  0  0 -1 -2 -2  0 -1 -2 -1  4  1 -3 -2 -2
 0 -1  0 -1 -1 -1 -1 -2 -2 -1 -1 -1 -1 -2 -1  1  5 -2 -2  0
-3 -3 -4 -4 -2 -2 -3 -2 -2 -3 -2 -3 -1  1 -4 -3 -2 11  2 -3
-2 -2 -2 -3 -2 -1 -2 -3  2 -1 -1 -2 -1  3 -3 -2 -2  2  7 -1
 0 -3 -3 -3 -1 -2 -2 -3 -3  3  1 -2  1 -1 -2 -2  0 -3 -1  4
""".strip().splitlines()], dtype=np.int8)
BACKGROUND = np.array([
    0.07805, 0.05129, 0.04487, 0.05364, 0.01925, 0.04264, 0.06295, 0.07377, 0.02199, 0.05142,
    0.09019, 0.05744, 0.02243, 0.03856, 0.05203, 0.07120, 0.05841, 0.01330, 0.03216, 0.06441])
# DNA: codes 0..3, +1 match, -3 mismatch, a gap of k bases costs 5 + 2k
DNA_MATRIX = np.full((20, 20), -3, dtype=np.int8)
np.fill_diagonal(DNA_MATRIX, 1)


def _search(db_n, q_n, q_lo, q_hi, mode, entry, sigma=0.5, homologs=0, gap_open=10, gap_extend=2):
    """A search: q_n queries of q_lo..q_hi residues (spread over the logarithm)
    against db_n proteins (median 300, 20..1000 residues) and `homologs`
    diverged copies of the longest query.  entry: "call" (one search() call,
    host queries to host scores) or "prepared" (a prepared batch, scores left
    on the device)."""
    return {"kind": "search", "db_n": db_n, "sigma": sigma, "homologs": homologs, "q_n": q_n, "q_lo": q_lo,
            "q_hi": q_hi, "gap_open": gap_open, "gap_extend": gap_extend, "mode": mode, "entry": entry}


def _pair(m, n):
    return {"kind": "pair", "m": m, "n": n}


def _trace(db_n, q_n, q_lo, q_hi, hits):
    """Alignments of each query's `hits` best hits (planted homologs of it)."""
    return {"kind": "trace", "db_n": db_n, "q_n": q_n, "q_lo": q_lo, "q_hi": q_hi, "hits": hits}


def listed():
    return [
        # an interactive lookup: one ordinary query against a small curated
        # set, through one call (planning, upload, search, download)
        dict(_search(2000, 1, 144, 144, "packed", "call"), name="one_query_2k"),
        # the same lookup repeated from a prepared batch, plain 32-bit cells
        dict(_search(2000, 1, 144, 144, "int32", "prepared"), name="one_query_2k_int32"),
        # many short queries (domains, peptides' parents) against the small set
        dict(_search(2000, 256, 144, 144, "packed", "prepared"), name="batch_256x144_2k"),
        # a very long protein and a short one against a set with close
        # relatives of the long one (scores past the 16-bit range), one call
        dict(_search(2000, 2, 144, 8000, "packed", "call", homologs=10), name="homologs_8k"),
        # the same with 32-bit cells, from a prepared batch
        dict(_search(2000, 2, 144, 8000, "int32", "prepared", homologs=10), name="homologs_8k_int32"),
        # a search server's batch: two arrived queries against a large
        # database with spread-out lengths, host to host
        dict(_search(500_000, 2, 353, 471, "packed", "call", sigma=0.65), name="serving_pair_500k"),
        # one long query against a mid-size database
        dict(_search(100_000, 1, 1301, 1301, "packed", "prepared"), name="single_query_100k"),
        # the protein benchmark: 20 queries of 144..5478 residues x 200,000
        dict(_search(200_000, 20, 144, 5478, "packed", "prepared"), name="twenty_queries_200k"),
        # the same queries with 32-bit cells against a tenth of the database
        dict(_search(20_000, 20, 144, 5478, "int32", "prepared"), name="twenty_queries_20k_int32"),
        # genome pairs: two short chromosomes / plasmids, two bacterial genomes
        dict(_pair(162_000, 172_000), name="dna_162k_172k"),
        dict(_pair(1_000_000, 1_000_000), name="dna_1m_1m"),
        # the alignments behind the best hits of a 20-query search
        dict(_trace(20_000, 20, 144, 5478, 10), name="traceback_200_hits"),
    ]


_LARGEST_CELLS = 2.0e12  # a drawn case stays within the largest listed search


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: small and large searches, DNA pairs, tracebacks; sizes
    uniform over their logarithm, so mostly odd and ragged."""
    kind = rng.choices(["small", "large", "pair", "trace"], [4, 4, 2, 1])[0]
    if kind == "pair":
        m = _log_int(rng, 20_000, 900_000)
        return _pair(m, max(20_000, min(1_000_000, int(m * rng.uniform(0.7, 1.4)))))
    if kind == "trace":
        lo = _log_int(rng, 60, 500)
        return _trace(_log_int(rng, 2000, 20_000), rng.randint(1, 20), lo, _log_int(rng, lo, 5000), rng.randint(1, 10))
    go, ge = rng.choice([(10, 2), (10, 2), (10, 1), (14, 2)])
    mode = rng.choice(["packed", "packed", "packed", "int32"])
    entry = rng.choice(["call", "prepared"])
    if kind == "small":
        q_n = _log_int(rng, 1, 200)
        lo = _log_int(rng, 20, 1000)
        hi = _log_int(rng, lo, 8000 if q_n < 5 else 2000) if q_n > 1 else lo
        homologs = rng.choice([0, 0, rng.randint(1, 12)])
        return _search(_log_int(rng, 300, 10_000), q_n, lo, hi, mode, entry, rng.choice([0.5, 0.65]), homologs, go, ge)
    db_n = _log_int(rng, 10_000, 300_000)
    lo = _log_int(rng, 40, 1500)
    q_n = _log_int(rng, 1, 60)
    hi = _log_int(rng, lo, 4000) if q_n > 1 else lo
    q_n = max(1, min(q_n, int(_LARGEST_CELLS / (3 if mode == "int32" else 1.5) / (db_n * 345.0 * hi))))
    return _search(db_n, q_n, lo, hi if q_n > 1 else lo, mode, entry, rng.choice([0.5, 0.65]), 0, go, ge)


# -- shapes (from the case alone) -------------------------------------------

def _query_lengths(case):
    n, lo, hi = case["q_n"], case["q_lo"], case["q_hi"]
    return [int(round(lo * (hi / lo) ** (k / max(1, n - 1)))) for k in range(n)]


def _db_lengths(n, sigma):
    z = np.random.Generator(np.random.PCG64(n)).standard_normal(n)
    return np.clip(np.rint(300.0 * np.exp(sigma * z)), 20, 1000).astype(np.int64)


# -- inputs (from the case and the seed) --------------------------------------

def _codes():
    """65536 residue codes in the background law's proportions."""
    edges = np.rint(np.cumsum(BACKGROUND) / BACKGROUND.sum() * 65536).astype(np.int64)
    return np.searchsorted(edges, np.arange(65536), side="right").clip(0, 19).astype(np.uint8)


def _residues(rng, total):
    return _codes()[rng.integers(0, 65536, size=int(total), dtype=np.uint16)]


def _diverged(rng, seq, fresh):
    """A copy of seq with 10 % substitutions and 1 % indel events (insertion or
    deletion, geometric lengths), cut or extended to seq's length; fresh(k)
    gives k random codes."""
    n = seq.size
    out = np.where(rng.random(n) < 0.10, fresh(n), seq)
    counts = np.ones(n, dtype=np.int64)
    event = rng.random(n) < 0.01
    insert = event & (rng.random(n) < 0.5)
    k = rng.geometric(0.5, size=n)
    for p in np.flatnonzero(event & ~insert):
        counts[p:p + k[p]] = 0
    counts[insert] += k[insert]
    at = np.cumsum(counts) - counts
    out = np.repeat(out, counts)
    extra = np.ones(out.size, dtype=bool)
    extra[at[counts > 0]] = False
    out[extra] = fresh(int(extra.sum()))
    if out.size < n:
        out = np.concatenate([out, fresh(n - out.size)])
    return np.ascontiguousarray(out[:n], dtype=np.uint8)


def _offsets(lengths):
    return np.concatenate([[0], np.cumsum(np.asarray(lengths, dtype=np.int64))]).astype(np.int64)


def _protein_inputs(case, seed):
    """(database residues, offsets, query residues, offsets, homolog positions)."""
    rng = np.random.Generator(np.random.PCG64(seed))
    q_off = _offsets(_query_lengths(case))
    q_res = _residues(rng, q_off[-1])
    lengths = _db_lengths(case["db_n"], case.get("sigma", 0.5))
    res = _residues(rng, lengths.sum())
    if case["kind"] == "trace":
        sources = [q for q in range(case["q_n"]) for _ in range(case["hits"])]
    else:
        sources = [case["q_n"] - 1] * case["homologs"]
    copies = [_diverged(rng, q_res[q_off[q]:q_off[q + 1]], lambda k: _residues(rng, k)) for q in sources]
    at = len(lengths) + np.arange(len(copies))  # (the database sorts by length itself)
    lengths = np.concatenate([lengths, [c.size for c in copies]]).astype(np.int64)
    return np.concatenate([res] + copies), _offsets(lengths), q_res, q_off, list(zip(sources, at.tolist()))


def _dna_inputs(case, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    fresh = lambda k: rng.integers(0, 4, size=k, dtype=np.uint8)  # noqa: E731
    target = fresh(case["n"])
    query = _diverged(rng, target[:min(case["m"], case["n"])], fresh)
    return np.concatenate([query, fresh(case["m"] - query.size)]), target


# -- the passes ----------------------------------------------------------------

def prepare(case, seed):
    if case["kind"] == "pair":
        query, target = _dna_inputs(case, seed)
        return {"kind": "pair", "query": query, "target": target}
    d_res, d_off, q_res, q_off, hits = _protein_inputs(case, seed)
    state = {"kind": case["kind"], "db": sw.Database(d_res, d_off), "q_res": q_res, "q_off": q_off, "hits": hits}
    state["path"] = 2 * max(_query_lengths(case))
    if case["kind"] == "search":
        state.update({k: case[k] for k in ("entry", "mode", "gap_open", "gap_extend")})
        if case["entry"] == "prepared":
            state["batch"] = sw.PreparedQueries(state["db"], q_res, q_off, BLOSUM62, case["gap_open"],
                                                case["gap_extend"], mode=case["mode"])
            state["out"] = torch.empty((case["q_n"], d_off.size - 1), dtype=torch.int32, device="cuda")
    return state


def run(state):
    if state["kind"] == "pair":
        return sw.align_pair(state["query"], state["target"], DNA_MATRIX, 5, 2)
    if state["kind"] == "trace":
        got = sw.traceback(state["db"], state["q_res"], state["q_off"], state["hits"], BLOSUM62)
        # (operations padded to the longest possible path, so that the shape depends on the case alone)
        return {"spans": np.array([a[:5] for a in got], dtype=np.int64),
                "ops": np.frombuffer("".join(a[5].ljust(state["path"], ".") for a in got).encode(), dtype=np.uint8)}
    if state["entry"] == "prepared":
        return state["batch"].search(state["out"])
    return sw.search(state["db"], state["q_res"], state["q_off"], BLOSUM62, state["gap_open"], state["gap_extend"],
                     mode=state["mode"])


def work(case):
    """Residues read and scores (or alignments) written once; the twelve
    operations of the recurrence per cell."""
    if case["kind"] == "pair":
        return {"bytes": case["m"] + case["n"] + 4, "flops": 12.0 * case["m"] * case["n"]}
    q_len = _query_lengths(case)
    if case["kind"] == "trace":
        cells = case["hits"] * sum(m * m for m in q_len)
        # (four direction bits per cell cannot be avoided without a second pass)
        return {"bytes": 3 * case["hits"] * sum(q_len) + cells / 2, "flops": 12.0 * cells}
    lengths = int(_db_lengths(case["db_n"], case["sigma"]).sum()) + case["homologs"] * q_len[-1]
    n = case["db_n"] + case["homologs"]
    return {"bytes": lengths + sum(q_len) + 4.0 * case["q_n"] * n, "flops": 12.0 * lengths * sum(q_len)}


# -- the scores from a plain 64-bit dynamic program -----------------------------

def _best(query, rows, matrix, go, ge):
    """Best local scores of one query against padded rows [B, n] (code 20
    past the end), anti-diagonal by anti-diagonal."""
    m, (b, n) = query.size, rows.shape
    dev = rows.device
    table = torch.full((20, 21), -(10 ** 6), dtype=torch.int64, device=dev)
    table[:, :20] = torch.as_tensor(matrix.astype(np.int64), device=dev)
    table = table.reshape(-1)
    base = torch.as_tensor(query.astype(np.int64), device=dev) * 21
    # column d - i of row i (1-based) on anti-diagonal d: a window of the reversed, padded rows
    pad = torch.full((b, m), 20, dtype=torch.int64, device=dev)
    rev = torch.cat([pad, rows.flip(1), pad], 1)
    h1 = torch.zeros((b, m + 1), dtype=torch.int64, device=dev)  # rows 0..m on the last anti-diagonal
    h2 = torch.zeros_like(h1)                                     # and on the one before
    e = torch.zeros_like(h1)
    f = torch.zeros_like(h1)
    best = torch.zeros((b, m), dtype=torch.int64, device=dev)
    for d in range(2, m + n + 1):
        s0 = m + n - d + 1
        s = table[base + rev[:, s0:s0 + m]]
        hg = h1 - go
        e = torch.maximum(hg, e - ge)
        f[:, 1:] = torch.maximum(hg[:, :-1], f[:, :-1] - ge)
        h = torch.maximum(h2[:, :-1] + s, torch.maximum(e[:, 1:], f[:, 1:])).clamp_(min=0)
        h2, h1 = h1, torch.cat([h1[:, :1], h], 1)
        torch.maximum(best, h, out=best)
    return best.amax(1)


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "pair":
        if case["m"] + case["n"] > 90_000:
            return None
        query, target = _dna_inputs(case, seed)
        rows = torch.as_tensor(target.astype(np.int64), device=dev)[None]
        return int(_best(query, rows, DNA_MATRIX, 7, 2)[0])
    if case["kind"] == "trace" or work(case)["flops"] > 12.0 * 8e9:
        return None
    d_res, d_off, q_res, q_off, _ = _protein_inputs(case, seed)
    lengths = np.diff(d_off)
    out = np.zeros((q_off.size - 1, lengths.size), dtype=np.int32)
    # the database in length-sorted groups, so that padding stays small
    order = np.argsort(lengths, kind="stable")
    cuts = [0] + [int(c) for c in np.searchsorted(lengths[order], [300, 1001], side="left")] + [lengths.size]
    for a, b in zip(cuts[:-1], cuts[1:]):
        ids = order[a:b]
        if not ids.size:
            continue
        rows = np.full((ids.size, int(lengths[ids].max())), 20, dtype=np.int64)
        for r, i in enumerate(ids):
            rows[r, :lengths[i]] = d_res[d_off[i]:d_off[i + 1]]
        rows = torch.as_tensor(rows, device=dev)
        for q in range(q_off.size - 1):
            got = _best(q_res[q_off[q]:q_off[q + 1]], rows, BLOSUM62, case["gap_open"] + case["gap_extend"],
                        case["gap_extend"])
            out[q, ids] = got.cpu().numpy()
    return torch.as_tensor(out)
