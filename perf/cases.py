"""Performance cases of the search framework: what a user's program has it do, through its public entry points.

A case is a dict of plain values. ``listed()`` names the standing ones, ``draw(rng)`` gives another one of the
same ranges, ``prepare(case, seed)`` makes inputs, index and plan, ``run(state)`` is one pass, ``exact(case,
seed)`` the same answer in 64 bits from plain torch, ``work(case)`` the bytes and operations of one pass.

Inputs are drawn on the GPU after the repository's synthetic workloads: document and query dims Zipf(s) without
replacement over a vocabulary of ``dim``, lognormal or uniform positive values, uneven row lengths.
"""
from __future__ import annotations

import math
import statistics

import numpy as np
import torch

import paper_2509_08395_gb300 as sindi

# Every field a case can have, with its default.
#   call      how the framework is called: "search" (device queries), "host" (numpy queries and results),
#             "plan" (a fixed batch replayed), "build" (documents on the device, index built and first asked),
#             "build_host" (the same from numpy documents)
#   docs, dim, zipf, values                documents; values "lognormal" (sigma 0.8) or "uniform"
#   nnz, nnz_sigma, nnz_min, nnz_max       row lengths of the documents: lognormal of that mean (sigma 0: fixed)
#   queries, q_nnz, q_sigma, q_min, q_max  the same for the queries; q_sigma < 0: uniform in [q_min, q_max]
#   window, alpha, dtype, prune, prune_n   the index
#   k, gamma, mode                         the search
_DEFAULTS = dict(call="search", docs=1_000_000, dim=30_522, zipf=1.05, values="lognormal", nnz=120.0,
                 nnz_sigma=0.5, nnz_min=10, nnz_max=400, queries=1_000, q_nnz=45.0, q_sigma=0.5, q_min=5, q_max=150,
                 window=16_384, alpha=0.5, dtype="f32", prune="mass", prune_n=0, k=50, gamma=500, mode="batched")


def _case(**kw) -> dict:
    return {**_DEFAULTS, **kw}


def listed() -> list:
    return [
        # one user's query at a time (interactive search, a retrieval step of an agent): latency
        _case(name="one-query", queries=1, k=10, gamma=200, mode="plain"),
        # a small collection searched exactly, unpruned and without a reorder: a per-tenant index, a test set
        _case(name="exact-10k", docs=10_000, dim=1_024, zipf=1.1, nnz=32.0, nnz_sigma=0.2, nnz_min=8, nnz_max=64,
              queries=100, q_nnz=8.0, q_sigma=0.35, q_min=1, q_max=32, window=4_096, alpha=1.0, k=10, gamma=0,
              mode="plain"),
        # a stream of independent queries over a passage collection of a million documents, one launch chain each
        _case(name="plain-1m", mode="plain"),
        # an offline job's batch over the same collection (evaluation runs, hard-negative mining)
        _case(name="batched-1m"),
        # a web service's micro-batch: queries and answers in host memory, a collection of an odd size, FP16 lists
        _case(name="host-64", call="host", docs=317_811, queries=61, dtype="f16", k=10, gamma=300),
        # a server's fixed micro-batch, recorded once and replayed
        _case(name="plan-32", call="plan", queries=32, dtype="f16"),
        # exact unpruned search of dense-ish uniform vectors (ground truth for recall, sparsity studies)
        _case(name="exact-uniform", zipf=0.0, dim=30_000, values="uniform", nnz=120.0, nnz_sigma=0.0, nnz_min=120,
              nnz_max=120, queries=200, q_nnz=120.0, q_sigma=0.0, q_min=120, q_max=120, alpha=1.0, gamma=0),
        # long uneven queries (expanded queries, documents as queries) with a deep pool, FP8 lists, default window
        _case(name="long-f8", docs=1_234_567, queries=500, q_sigma=-1.0, q_nnz=102.5, q_min=5, q_max=200,
              window=8_192, dtype="f8", k=100, gamma=2_000),
        # a full passage collection, FP16 lists, a deep reorder: the largest
        _case(name="large-f16", docs=8_800_000, window=8_192, dtype="f16", gamma=1_000),
        # the collection is indexed again (new documents, a new encoder) and answers its first batch
        _case(name="build-1m", call="build", queries=16),
        # a ragged collection (a few documents of thousands of entries) indexed from host arrays, lists cut too, FP8
        _case(name="build-ragged", call="build_host", docs=100_003, dim=50_021, nnz=96.0, nnz_sigma=1.1, nnz_min=1,
              nnz_max=3_000, queries=16, window=8_192, alpha=0.7, dtype="f8", prune="mass_list", prune_n=3_000,
              k=10, gamma=200),
    ]


def _log_int(rng, lo: int, hi: int) -> int:
    return max(lo, min(hi, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng) -> dict:
    call = rng.choice(("search", "search", "search", "host", "plan", "build", "build_host"))
    docs = _log_int(rng, 10_000, 200_000 if call == "build_host" else 2_000_000)
    dim = _log_int(rng, 1_024, 100_003)
    k = _log_int(rng, 1, 200)
    exact_search = call == "search" and rng.random() < 0.3
    gamma = 0 if exact_search else _log_int(rng, max(k, 50), 2_500)
    queries = {"build": 16, "build_host": 16, "plan": _log_int(rng, 1, 256), "host": _log_int(rng, 1, 256),
               "search": _log_int(rng, 1, 200 if exact_search else 1_000)}[call]
    nnz = float(min(_log_int(rng, 24, 140), dim // 8))
    q_mean = float(min(_log_int(rng, 4, 120), dim // 8))
    prune = rng.choice(("mass", "mass", "vector_number", "mass_list")) if call.startswith("build") else "mass"
    case = _case(call=call, docs=docs, dim=dim, zipf=rng.choice((0.0, 1.0, 1.05, 1.1)),
                 values=rng.choice(("lognormal", "lognormal", "uniform")), nnz=nnz,
                 nnz_sigma=rng.choice((0.3, 0.5, 0.9)), nnz_min=1, nnz_max=int(4 * nnz), queries=queries, q_nnz=q_mean,
                 q_sigma=rng.choice((0.3, 0.5, -1.0)), q_min=1, q_max=int(2 * q_mean),
                 window=rng.choice((2_048, 4_096, 8_192, 10_000, 16_384, 32_768)),
                 alpha=1.0 if exact_search else rng.choice((0.4, 0.5, 0.7, 1.0)), dtype=rng.choice(("f32", "f16", "f8")),
                 prune=prune, prune_n={"mass": 0, "vector_number": 25, "mass_list": 4_000}[prune], k=k, gamma=gamma,
                 mode="batched" if call in ("plan", "host") else rng.choice(("plain", "batched")))
    while case["queries"] > 1 and work(case)["flops"] > 1.2e10:  # well below the largest listed one
        case["queries"] //= 2
    return case


# ---- inputs -----------------------------------------------------------------------------------------------
def _zipf_probs(dim: int, s: float, device=None):
    p = torch.arange(1, dim + 1, dtype=torch.float64, device=device).pow(-s)
    return p / p.sum()


def _row_lengths(n: int, mean: float, sigma: float, lo: int, hi: int, g):
    if sigma < 0:  # uniform
        return torch.randint(lo, hi + 1, (n,), generator=g, device="cuda")
    z = torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    return torch.exp(math.log(mean) - 0.5 * sigma * sigma + sigma * z).round().long().clamp_(lo, hi)


def _rows(n: int, dim: int, zipf: float, values: str, lengths, g):
    """CSR rows of distinct dims, ascending in a row: draws from Zipf(s) until the row's length is reached (rows
    whose spare draws run out end a little shorter)."""
    cdf = _zipf_probs(dim, zipf, "cuda").cumsum(0) if zipf > 0 else None
    counts, dims, vals = [], [], []
    step = 1_000_000
    for r0 in range(0, n, step):
        want = lengths[r0:r0 + step].clamp(max=dim)
        m = want.numel()
        tries = (want.double() * (1.6 if zipf > 0 else 1.1)).long() + 12
        first = torch.zeros(m + 1, dtype=torch.long, device="cuda")
        torch.cumsum(tries, 0, out=first[1:])
        total = int(first[-1])
        row = torch.repeat_interleave(torch.arange(m, device="cuda"), tries, output_size=total)
        u = torch.rand(total, generator=g, device="cuda", dtype=torch.float64)
        d = torch.searchsorted(cdf, u).clamp_(max=dim - 1) if zipf > 0 else (u * dim).long().clamp_(max=dim - 1)
        del u
        key, perm = torch.sort(row * dim + d, stable=True)
        del d
        new = torch.ones(total, dtype=torch.bool, device="cuda")
        new[1:] = key[1:] != key[:-1]
        fresh = torch.zeros(total, dtype=torch.int32, device="cuda")
        fresh[perm[new]] = 1  # a dim's first draw in its row
        seen = torch.cumsum(fresh, 0, dtype=torch.int32)  # of the chunk's rows up to here
        before = (seen - fresh)[first[:-1]]
        keep = new & ((seen[perm] - before[row[perm]]) <= want[row[perm]])
        del new, fresh, seen, perm
        key = key[keep]
        del keep
        rr = key // dim
        counts.append(torch.bincount(rr, minlength=m))
        dims.append((key - rr * dim).int())
        del rr, key
        x = dims[-1].numel()
        if values == "uniform":
            vals.append(1.0 - torch.rand(x, generator=g, device="cuda"))
        else:
            vals.append(torch.exp(0.8 * torch.randn(x, generator=g, device="cuda")))
    indptr = torch.zeros(n + 1, dtype=torch.long, device="cuda")
    torch.cumsum(torch.cat(counts), 0, out=indptr[1:])
    return indptr, torch.cat(dims), torch.cat(vals)


def _inputs(case: dict, seed: int):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    c = case
    docs = _rows(c["docs"], c["dim"], c["zipf"], c["values"],
                 _row_lengths(c["docs"], c["nnz"], c["nnz_sigma"], c["nnz_min"], c["nnz_max"], g), g)
    queries = _rows(c["queries"], c["dim"], c["zipf"], c["values"],
                    _row_lengths(c["queries"], c["q_nnz"], c["q_sigma"], c["q_min"], c["q_max"], g), g)
    return docs, queries


def _build(case: dict, docs):
    return sindi.Index(*docs, case["dim"], window=case["window"], alpha=case["alpha"], value_dtype=case["dtype"],
                       prune=case["prune"], prune_n=case["prune_n"])


# ---- one pass ---------------------------------------------------------------------------------------------
def prepare(case: dict, seed: int):
    docs, queries = _inputs(case, seed)
    st = {"case": case, "queries": queries}
    if case["call"] == "build":
        st["docs"] = docs
    elif case["call"] == "build_host":
        st["docs"] = tuple(t.cpu().numpy() for t in docs)
    else:
        st["index"] = _build(case, docs)
        if case["call"] == "host":
            st["queries"] = tuple(t.cpu().numpy() for t in queries)
        elif case["call"] == "plan":
            st["plan"] = sindi.Plan(st["index"], *queries, k=case["k"], gamma=case["gamma"])
        else:  # a program that searches again and again keeps its result buffers
            shape = (case["queries"], case["k"])
            st["out"] = (torch.empty(shape, dtype=torch.int32, device="cuda"),
                         torch.empty(shape, dtype=torch.float32, device="cuda"))
    return st


def run(state):
    c = state["case"]
    if c["call"] == "plan":
        return state["plan"].launch()
    if c["call"].startswith("build"):
        with _build(c, state["docs"]) as idx:
            ids, scores = idx.search(*state["queries"], k=c["k"], gamma=c["gamma"], mode=c["mode"])
            return ids, scores, idx.info["postings"]
    return state["index"].search(*state["queries"], k=c["k"], gamma=c["gamma"], mode=c["mode"], out=state.get("out"))


# ---- the same in 64 bits ----------------------------------------------------------------------------------
def _csr(indptr, dims, vals, dim: int):
    return torch.sparse_csr_tensor(indptr.int(), dims.int(), vals, size=(indptr.numel() - 1, dim), dtype=torch.float64)


def _kept(case: dict, docs):
    """Which entries of the documents become postings (64-bit sums over |x| descending, lower dim first)."""
    indptr, dims, vals = docs
    n = indptr.numel() - 1
    keep = torch.ones(dims.numel(), dtype=torch.bool, device="cuda")
    for r0 in range(0, n, 1_000_000):  # row rule
        r1 = min(n, r0 + 1_000_000)
        b, e = int(indptr[r0]), int(indptr[r1])
        if e == b or (case["alpha"] >= 1.0 and case["prune"] != "vector_number"):
            continue
        start = indptr[r0:r1] - b
        row = torch.repeat_interleave(torch.arange(r1 - r0, device="cuda"), indptr[r0 + 1:r1 + 1] - indptr[r0:r1])
        by_value = torch.sort(vals[b:e].abs(), descending=True, stable=True).indices
        order = by_value[torch.sort(row[by_value], stable=True).indices]  # rows in order, |x| descending in a row
        rank = torch.arange(e - b, device="cuda") - start[row]
        if case["prune"] == "vector_number":
            good = rank < case["prune_n"]
        else:
            a = vals[b:e].abs().double()
            mass = torch.zeros(r1 - r0, dtype=torch.float64, device="cuda").index_add_(0, row, a)
            run_sum = a[order].cumsum(0)
            before = run_sum - a[order]
            before = before - before[start.clamp(max=e - b - 1)][row]
            good = before < case["alpha"] * mass[row]
        keep[b:e] = False
        keep[b + order[good]] = True
    if case["prune"] in ("list", "mass_list"):  # the largest entries of every list, lower document first
        at = keep.nonzero().squeeze(1)
        by_value = torch.sort(vals[at].abs(), descending=True, stable=True).indices
        order = by_value[torch.sort(dims[at][by_value], stable=True).indices]
        cnt = torch.bincount(dims[at].long(), minlength=case["dim"])
        first = cnt.cumsum(0) - cnt
        rank = torch.arange(at.numel(), device="cuda") - first[dims[at][order].long()]
        keep[at[order[rank >= case["prune_n"]]]] = False
    return keep


def _stored(case: dict, dims, vals):
    """The value a posting stores, in its type."""
    if case["dtype"] == "f16":
        return vals.half().float()
    if case["dtype"] == "f8":
        top = torch.zeros(case["dim"], device="cuda").scatter_reduce_(0, dims.long(), vals.abs(), "amax")
        scale = top / 448.0
        scale = torch.where(scale > 0, scale, torch.ones_like(scale))[dims.long()]
        return ((vals / scale).to(torch.float8_e4m3fn).float().double() * scale.double())
    return vals


def exact(case: dict, seed: int):
    docs, queries = _inputs(case, seed)
    indptr, dims, vals = docs
    keep = _kept(case, docs)
    n, nq, k = case["docs"], case["queries"], case["k"]
    pool = min(case["gamma"] or k, n)
    row_kept = torch.zeros(n + 1, dtype=torch.long, device="cuda")
    row_kept[1:] = torch.cumsum(keep, 0)[indptr[1:] - 1] * (indptr[1:] > 0)
    kdims = dims[keep]
    kvals = _stored(case, kdims, vals[keep])
    del keep
    out = torch.empty((nq, k), dtype=torch.float64, device="cuda")
    qp, qd, qv = queries
    for q0 in range(0, nq, 128):
        q1 = min(nq, q0 + 128)
        b, e = int(qp[q0]), int(qp[q1])
        Q = torch.zeros((case["dim"], q1 - q0), dtype=torch.float64, device="cuda")
        col = torch.repeat_interleave(torch.arange(q1 - q0, device="cuda"), qp[q0 + 1:q1 + 1] - qp[q0:q1])
        Q[qd[b:e].long(), col] = qv[b:e].double()
        coarse, full = [], []
        for r0 in range(0, n, 1_000_000):  # the best of every block of documents, then of all
            r1 = min(n, r0 + 1_000_000)
            kb, ke = int(row_kept[r0]), int(row_kept[r1])
            top = (_csr(row_kept[r0:r1 + 1] - kb, kdims[kb:ke], kvals[kb:ke].double(), case["dim"]) @ Q).t().contiguous()
            c, at = torch.topk(top, min(pool, r1 - r0), dim=1)
            coarse.append(c)
            if case["gamma"]:
                b, e = int(indptr[r0]), int(indptr[r1])
                x = _csr(indptr[r0:r1 + 1] - b, dims[b:e], vals[b:e].double(), case["dim"]) @ Q
                full.append(torch.gather(x.t(), 1, at))
            del top
        coarse = torch.cat(coarse, 1)
        best, at = torch.topk(coarse, pool, dim=1)
        if case["gamma"]:
            best = torch.gather(torch.cat(full, 1), 1, at)
        best = torch.topk(best, min(k, pool), dim=1).values
        out[q0:q1] = -math.inf
        out[q0:q1, :best.shape[1]] = best
    if case["call"] == "host":
        return None, out.cpu().numpy()
    if case["call"].startswith("build"):
        return None, out, int(row_kept[-1])
    return None, out


# ---- bytes and operations ---------------------------------------------------------------------------------
def _inclusion(dim: int, s: float, mean: float) -> np.ndarray:
    """The share of rows that hold each dim, for rows of `mean` distinct Zipf(s) dims."""
    p = np.arange(1, dim + 1, dtype=np.float64) ** -s
    p /= p.sum()
    lo, hi = 0.0, 1e9
    for _ in range(80):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if -np.expm1(-mid * p).sum() < mean else (lo, mid)
    return -np.expm1(-hi * p)


def _kept_share(case: dict) -> float:
    """The share of the documents' entries that become postings (before list pruning)."""
    if case["prune"] == "vector_number":
        return min(1.0, case["prune_n"] / case["nnz"])
    if case["alpha"] >= 1.0:
        return 1.0
    if case["values"] == "uniform":
        return 1.0 - math.sqrt(1.0 - case["alpha"])
    nd = statistics.NormalDist()
    return 1.0 - nd.cdf(0.8 + nd.inv_cdf(1.0 - case["alpha"]))


def work(case: dict) -> dict:
    """Searches: the posting lists of the queries' terms (each list once), the queries, one document row per
    reorder candidate (each row at most once), the results; two operations per posting and query, two per entry of a
    reordered row. Builds: the documents read, the index (lists, offsets, the documents it keeps) written, too."""
    c = case
    vbytes = {"f32": 4, "f16": 2, "f8": 1}[c["dtype"]]
    lists = c["docs"] * _inclusion(c["dim"], c["zipf"], c["nnz"]) * _kept_share(c)
    if c["prune"] in ("list", "mass_list"):
        lists = np.minimum(lists, c["prune_n"])
    holds = _inclusion(c["dim"], c["zipf"], c["q_nnz"])
    touched = float((lists * holds).sum()) * c["queries"]
    union = float((lists * -np.expm1(c["queries"] * np.log1p(-np.minimum(holds, 1 - 1e-12)))).sum())
    rows = min(c["docs"], c["queries"] * min(c["gamma"], c["docs"]))
    pool = c["queries"] * min(c["gamma"], c["docs"])
    doc_bytes = c["docs"] * (8 * c["nnz"] + 8)
    b = union * (2 + vbytes) + c["queries"] * (8 * c["q_nnz"] + 8) + rows * 8 * c["nnz"] + c["queries"] * c["k"] * 8
    f = 2 * touched + 2 * pool * c["nnz"]
    if c["call"].startswith("build"):
        sigma = -(-c["docs"] // c["window"])
        b += 2 * doc_bytes + float(lists.sum()) * (2 + vbytes) + 4 * c["dim"] * sigma
        f += c["docs"] * c["nnz"]
    return {"bytes": float(b), "flops": float(f)}
