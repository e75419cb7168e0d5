"""The work that users of this framework have it do, as measurable cases.

Every case goes through a public entry point of ``paper_2602_17099_gb300.rnsm``:
whole merges (the product), segment builds, query searches, and the prune and
reverse-edge calls that an index maintainer makes by themselves.  Sizes,
dimensions, degrees and beams are those of this repository's workloads and
tests or lie between them; the rows come from the same recipes (SIFT-like
integers, DEEP-like and embedding-like unit vectors, plain Gaussians), drawn on
the device so that inputs can be made anew from a seed in a moment.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_2602_17099_gb300 import rnsm

_PREC = {"fp32": rnsm.FP32, "bf16": rnsm.BF16, "fp8": rnsm.FP8}
_DIM = {"sift": 128, "deep": 96, "embed": 768, "gauss": 32}
_CHUNK = 1 << 14


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the headline: two halves of a SIFT-sized index become one
        _merge("merge_sift_2x500k_fp32", "sift", 1_000_000, 2, 32, 64, "fp32"),
        # a sharded build: uneven cluster partitions, merged in MOS order
        _merge("merge_deep_mos5_bf16", "deep", 300_007, 5, 32, 64, "bf16", uneven=True),
        # text / image embeddings: inner product, wide rows, high degree
        _merge("merge_embed_3x20k_fp8", "embed", 60_000, 3, 64, 128, "fp8"),
        # the smallest merge: a fresh in-memory segment flushed into another
        _merge("merge_gauss_2x5k_fp32", "gauss", 10_000, 2, 16, 32, "fp32"),
        # incremental indexing: a day's new rows merged into a standing index
        {**_merge("merge_deep_increment_fp32", "deep", 158_001, 2, 32, 64, "fp32"),
         "increment": 8_001},
        # a segment's graph built from its rows
        {"name": "build_deep_60k", "kind": "build", "recipe": "deep", "n": 60_000, "R": 32,
         "L": 64},
        # a batch of queries against a standing index
        _search("search_sift_batch", "sift", 200_000, 10_000, 32, 64, 10),
        # online queries: a handful at a time, latency counts
        _search("search_deep_online", "deep", 100_003, 16, 32, 128, 10),
        # neighbour lists re-pruned after an update: ragged pools, FP32
        _prune("prune_deep_ragged_fp32", "deep", 100_001, 100_001, 32, 64, "fp32"),
        # the same on embeddings: wide pools, tensor-core tiles
        _prune("prune_embed_wide_bf16", "embed", 16_000, 16_000, 64, 128, "bf16"),
        # a few owners from a service that lets no library allocate
        {**_prune("prune_noalloc_small", "gauss", 4_000, 75, 16, 48, "fp32"), "noalloc": True},
        # back edges of new links entered into standing lists
        {"name": "reverse_edges_deep", "kind": "reverse", "recipe": "deep", "n": 150_000, "R": 32,
         "per_vertex": 11},
    ]


def draw(rng: random.Random):
    """One more case: a kind by its share of the listed ones, sizes spread over
    their range on a log scale, odd values among them."""
    kind = rng.choice(["merge", "merge", "merge", "build", "search", "search", "prune", "prune",
                       "noalloc", "reverse"])
    recipe = rng.choice(["sift", "deep", "deep", "embed", "gauss"])
    wide = recipe == "embed"
    R = rng.choice([48, 64]) if wide else rng.choice([16, 24, 32])
    L = rng.choice([64, 96, 128]) if wide else rng.choice([32, 48, 64])
    prec = rng.choice(["fp32", "fp32", "bf16", "fp8"])
    top = 60_000 if wide else 500_000
    if kind == "merge":
        total = _spread(rng, 4_000, top)
        m = rng.choice([2, 2, 3, 4, 6])
        c = _merge("", recipe, total, m, R, L, prec, uneven=rng.random() < 0.5)
        if m == 2 and rng.random() < 0.4:
            c["increment"] = max(500, int(total * rng.uniform(0.02, 0.3)))
    elif kind == "build":
        c = {"kind": "build", "recipe": recipe, "n": _spread(rng, 2_000, top // 4), "R": R, "L": L}
    elif kind == "search":
        ef = rng.choice([16, 32, 50, 64, 100, 128])
        c = _search("", recipe, _spread(rng, 5_000, top // 2), _spread(rng, 1, 20_000), R, ef,
                    rng.choice([1, 10, 10, min(ef, 16)]))
    elif kind == "prune":
        n = _spread(rng, 2_000, top // 3)
        pool = rng.randint(R + 1, 2 * R)
        c = _prune("", recipe, n, rng.randint(n // 4, n), R, pool, prec)
    elif kind == "noalloc":
        n = _spread(rng, 2_000, 50_000)
        c = {**_prune("", recipe, n, _spread(rng, 16, min(n, 4_000)), R, rng.randint(R, 2 * R),
                      "fp32"), "noalloc": True}
    else:
        c = {"kind": "reverse", "recipe": recipe, "n": _spread(rng, 3_000, top // 3), "R": R,
             "per_vertex": rng.randint(2, 20)}
    c.pop("name", None)
    return c


def _merge(name, recipe, total, m, R, L, prec, uneven=False):
    return {"name": name, "kind": "merge", "recipe": recipe, "total": total, "m": m, "R": R,
            "L": L, "prec": prec, "uneven": uneven, "increment": 0}


def _search(name, recipe, n, nq, R, ef, k):
    return {"name": name, "kind": "search", "recipe": recipe, "n": n, "nq": nq, "R": R, "ef": ef,
            "k": k}


def _prune(name, recipe, n, owners, R, pool, prec):
    return {"name": name, "kind": "prune", "recipe": recipe, "n": n, "owners": owners, "R": R,
            "pool": pool, "prec": prec, "noalloc": False}


def _spread(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _metric(case):
    return rnsm.IP if case["recipe"] == "embed" else rnsm.L2


def _sizes(case):
    total, m = case["total"], case["m"]
    if case["increment"]:
        return [case["increment"], total - case["increment"]]
    if case["uneven"]:
        w = [math.exp(0.6 * math.sin(2.4 * j + 1.0)) for j in range(m)]   # about 1 : 3
    else:
        w = [1.0] * m
    cut = [int(round(total * sum(w[:j]) / sum(w))) for j in range(m + 1)]
    return [cut[j + 1] - cut[j] for j in range(m)]


# -------------------------------------------------------------------- inputs

def _rows(recipe, n, seed, by_cluster=False):
    """n rows of a recipe on the device, all from the seed.  A mixture of
    low-rank Gaussian clusters (rank 32: the local intrinsic dimensionality of
    the real sets), as in workloads/generators.py; with by_cluster the rows are
    ordered by cluster, so that consecutive slices are cluster partitions."""
    d = _DIM[recipe]
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    kw = dict(generator=g, device="cuda", dtype=torch.float32)
    if recipe == "gauss":
        return torch.randn(n, d, **kw)
    n_comp = max(1, min(1000, n // 50))
    rank = 32
    if recipe == "sift":
        mean, spread, noise = torch.rand(n_comp, d, **kw) * 128.0, 4.0, 3.0
        A = torch.randn(n_comp, d, rank, **kw) * spread
    else:
        mean = torch.nn.functional.normalize(torch.randn(n_comp, d, **kw), dim=1)
        A = torch.randn(n_comp, d, rank, **kw)
        if recipe == "deep":
            A, noise = A * 0.06, 0.01
        else:   # near-orthonormal columns with falling singular values
            sv = 0.3 * 0.9 ** torch.arange(rank, device="cuda", dtype=torch.float32)
            A, noise = A * (sv / math.sqrt(d)), 0.013
    comp = torch.randint(0, n_comp, (n,), generator=g, device="cuda")
    comp, _ = torch.sort(comp)
    x = torch.empty(n, d, device="cuda")
    for s in range(0, n, _CHUNK):
        c = comp[s:s + _CHUNK]
        z = torch.randn(c.numel(), rank, 1, **kw)
        x[s:s + _CHUNK] = mean[c] + torch.bmm(A[c], z).squeeze(2)
        x[s:s + _CHUNK] += noise * torch.randn(c.numel(), d, **kw)
    if recipe == "sift":
        x = x.round_().clamp_(0.0, 255.0)
    else:
        x = torch.nn.functional.normalize(x, dim=1)
    if by_cluster:
        return x
    return x[torch.randperm(n, generator=g, device="cuda")].contiguous()


def prepare(case, seed):
    kind, recipe, R = case["kind"], case["recipe"], case["R"]
    metric = _metric(case)
    st = {"case": case, "metric": metric}
    if kind == "merge":
        sizes = _sizes(case)
        # random halves are the paper's first setting, cluster partitions its second
        x = _rows(recipe, case["total"], seed, by_cluster=case["uneven"])
        segs = []
        for s in torch.split(x, sizes):
            v = s.clone()
            adj, entry = rnsm.build_segment(v, R, case["L"], 1.2, metric)
            segs.append((v, adj, entry))
        st["segs"] = segs
        st["params"] = rnsm.params(R, case["L"], 1.2, metric, _PREC[case["prec"]])
        st["sizes"] = sizes
        st["centroids"] = np.stack([v.mean(dim=0).cpu().numpy() for v, _, _ in segs])
        return st
    if kind == "build":
        st["x"] = _rows(recipe, case["n"], seed)
        return st
    extra = case["nq"] if kind == "search" else 0
    x = _rows(recipe, case["n"] + extra, seed)
    st["x"] = x[:case["n"]].clone()
    st["adj"], entry = rnsm.build_segment(st["x"], R, 2 * R, 1.2, metric)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + 1)
    if kind == "search":
        st["q"] = x[case["n"]:].clone()
        st["seeds"] = torch.full((extra, 1), entry, dtype=torch.int32, device="cuda")
    elif kind == "prune":
        # the owner's list and the lists of its first neighbours, as an update
        # would gather them: repeats, the owner itself and -1 holes among them
        own = torch.randperm(case["n"], generator=g, device="cuda")[:case["owners"]].sort()[0]
        adj = st["adj"].long()
        lists = [adj[own], adj[adj[own, 0].clamp_min(0)], adj[adj[own, 1].clamp_min(0)]]
        st["pool"] = torch.cat(lists, 1)[:, :case["pool"]].to(torch.int32).contiguous()
        st["owners"] = own.to(torch.int32)
    else:
        # new links v -> u to vertices two steps away; u gains v
        adj = st["adj"].long()
        v = torch.arange(case["n"], device="cuda").repeat_interleave(case["per_vertex"])
        j = torch.randint(0, R, (2, v.numel()), generator=g, device="cuda")
        u = adj[v, j[0]]
        u = adj[u.clamp_min(0), j[1]]
        ok = (u >= 0) & (u != v)
        st["eu"], st["ev"] = u[ok].to(torch.int32), v[ok].to(torch.int32)
    return st


# ---------------------------------------------------------------------- runs

def run(st):
    case = st["case"]
    kind, R, metric = case["kind"], case["R"], st["metric"]
    if kind == "merge":
        plan = rnsm.mos_plan(st["sizes"], st["centroids"]) if case["m"] > 2 else None
        merged, _ = rnsm.merge(st["segs"], st["params"], plan)
        return merged
    if kind == "build":
        adj, entry = rnsm.build_segment(st["x"], R, case["L"], 1.2, metric)
        return adj, entry
    if kind == "search":
        ids, dists, _ = rnsm.search(st["x"], st["adj"], st["q"], st["seeds"], case["ef"],
                                    case["k"], metric)
        return ids, dists
    if kind == "prune":
        if case["noalloc"]:
            return rnsm.prune_noalloc(st["x"], st["owners"], st["pool"], R, 1.2, metric)
        return rnsm.prune(st["x"], st["owners"], st["pool"], R, 1.2, metric,
                          prec=_PREC[case["prec"]])
    # the caller keeps the lists as they were (readers still use them)
    return rnsm.reverse_edges(st["x"], st["adj"].clone(), st["eu"], st["ev"], 1.2, metric)


def work(case):
    """Bytes: inputs once, outputs once.  Operations: 2 * d per inner-product and
    3 * d per L2 distance; a beam search evaluates about 12 vertices per beam
    entry on these graphs, a prune every candidate against its owner and about a
    quarter of the candidate pairs."""
    kind, R, d = case["kind"], case["R"], _DIM[case["recipe"]]
    per = d * (2 if case["recipe"] == "embed" else 3)
    if kind == "merge":
        n, L = case["total"], case["L"]
        src = case["increment"] or n - n // case["m"]
        ndc = src * (12 * 17 + 12 * (L + 4 * ((L + 1) // 2)) // 5)
        pool = R + (L + 1) // 2
        ndc += 2 * src * (pool + pool * pool // 8)
        return {"bytes": n * (4 * d + 8 * R), "flops": ndc * per}
    if kind == "build":
        n, L = case["n"], case["L"]
        return {"bytes": n * (4 * d + 4 * R), "flops": n * (12 * L + L + L * L // 8) * per}
    if kind == "search":
        n, nq = case["n"], case["nq"]
        # rows and lists that the beams touch at least once, at most the whole index
        seen = min(n, nq * 12 * case["ef"])
        out = nq * (4 * d + 4 + 8 * case["k"])
        return {"bytes": seen * 4 * d + min(n, nq * case["ef"]) * 4 * R + out,
                "flops": nq * 12 * case["ef"] * per}
    if kind == "prune":
        nv, w = case["owners"], case["pool"]
        rows = min(case["n"], nv * (w + 1))
        return {"bytes": rows * 4 * d + nv * 4 * (1 + w + R), "flops": nv * (w + w * w // 8) * per}
    n, e = case["n"], case["n"] * case["per_vertex"]
    w = R + case["per_vertex"]
    return {"bytes": n * (4 * d + 8 * R) + 8 * e, "flops": n * (w + w * w // 8) * per}


# --------------------------------------------------------------------- exact

def exact(case, seed):
    """Searches return distances: the beam search of Algorithm 1 in 64 bits.  All
    other outputs are ids."""
    if case["kind"] != "search" or case["nq"] * case["n"] > 4_000_000_000:
        return None
    st = prepare(case, seed)
    x, adj, q = st["x"].double(), st["adj"].long(), st["q"].double()
    n, nq, ef, k, R = case["n"], case["nq"], case["ef"], case["k"], case["R"]
    qb = max(1, min(nq, 1_000_000_000 // n))   # queries at a time (a visited table of bytes)
    out = []
    for s in range(0, nq, qb):
        qs = q[s:s + qb]
        b = qs.shape[0]
        row = torch.arange(b, device="cuda")

        def dist(ids):
            r = x[ids.clamp_min(0)]
            if st["metric"] == rnsm.IP:
                return 1.0 - (r * qs[:, None, :]).sum(-1)
            return ((r - qs[:, None, :]) ** 2).sum(-1)

        seen = torch.zeros(b, n, dtype=torch.bool, device="cuda")
        start = st["seeds"][s:s + qb].long()
        ids = torch.full((b, ef), -1, dtype=torch.int64, device="cuda")
        dd = torch.full((b, ef), math.inf, dtype=torch.float64, device="cuda")
        done = torch.ones(b, ef, dtype=torch.bool, device="cuda")
        ids[:, :1], dd[:, :1], done[:, 0] = start, dist(start), False
        seen[row, start[:, 0]] = True
        while True:
            has, pick = (~done).max(dim=1)     # the first open entry: nearest
            if not bool(has.any()):
                break
            cur = ids[row, pick]
            done[row, pick] = True
            nb = torch.where(has[:, None], adj[cur.clamp_min(0)], -1)
            new = (nb >= 0) & ~seen[row[:, None], nb.clamp_min(0)]
            seen[row[:, None].expand(b, R)[new], nb[new]] = True
            nd = torch.where(new, dist(nb), math.inf)
            ci, cd = torch.cat([ids, nb], 1), torch.cat([dd, nd], 1)
            cf = torch.cat([done, ~new], 1)
            o = torch.argsort(ci, dim=1, stable=True)   # ties in distance: lower id first
            o = o.gather(1, torch.argsort(cd.gather(1, o), dim=1, stable=True))[:, :ef]
            ids, dd, done = ci.gather(1, o), cd.gather(1, o), cf.gather(1, o)
        out.append(dd[:, :k])
    return [None, torch.cat(out)]
