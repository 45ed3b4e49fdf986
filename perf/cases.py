"""Performance cases: the work that users of the library have it do, through the public binding.

Every case is a dict of plain values with a ``kind``:

* ``sign``     -- minhash_sign of an uploaded polygon set (A1), with or without the stream index;
* ``ingest``   -- a database step: poly_reload, minhash_sign, lsh_rebuild, and a few queries joined
                  against the rebuilt index (A0-A4);
* ``hashmap``  -- lsh_query on a single hashmap keyed on all K hashes (the paper's own setting);
* ``shortlist``-- a query batch's plain calls between signing and refinement: lsh_query,
                  jaccard_estimate with band bits, topm (A4-A6);
* ``search``   -- one replay of the captured query graph, plain or with the learned reranker;
* ``truth``    -- the exhaustive exact search: bbox_join and pair_jaccard of every pair (A8);
* ``refine``   -- pair_jaccard of given pairs of coastline-like polygons (A8);
* ``score``    -- reranker forward pass on feature rows and the top-m by score (A7, A6);
* ``gradients``-- one training batch of the reranker, forward and backward (A7).

Polygons, sizes, K, bands and area fractions are those of the named workloads, the tests and the
benchmark (or lie inside their ranges).  Inputs are drawn from the seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2511_16576_gb300 import binding as B
from paper_2511_16576_gb300 import synth

SEED, LSH_SEED, T24 = 0x5EED, 0x15A, 1 << 24

# polygon families: vertex-count range, distribution, area fractions, outline
_SHAPES = {
    "small": dict(n_range=(8, 64), n_dist="uniform", f_range=(1e-2, 5e-2)),
    "scale": dict(n_range=(16, 256), n_dist="loguniform", f_range=(1e-4, 1e-2)),
    "combined": dict(n_range=(8, 1024), n_dist="loguniform", f_range=(1e-5, 1e-2), fractal=True,
                     comonotone=True),
    "coastline": dict(n_range=(4, 65536), n_dist="loguniform", f_range=(1e-5, 1e-1), fractal=True,
                      comonotone=True),
}


def listed():
    return [
        # the smallest configuration as a first user runs it: no stream index, latency-bound
        {"name": "sign_small", "kind": "sign", "shape": "small", "polys": 1000, "max_verts": 0, "K": 32,
         "index": False},
        # signing a database of plain star polygons, K = 128, through the stream index
        {"name": "sign_scale", "kind": "sign", "shape": "scale", "polys": 300_000, "max_verts": 0,
         "K": 128, "index": True},
        # a few thousand coastline-like polygons of very uneven size, up to 65,536 vertices
        {"name": "sign_coastline", "kind": "sign", "shape": "coastline", "polys": 8000, "max_verts": 0,
         "K": 256, "index": True},
        # the database part of the benchmark's step on a slice of its workload
        {"name": "ingest_combined", "kind": "ingest", "shape": "combined", "polys": 400_000, "K": 128,
         "bands": 16, "queries": 256},
        # the paper's search on the 149,000-polygon centred set: one hashmap keyed on three hashes
        {"name": "hashmap_paper", "kind": "hashmap", "polys": 149_000, "mean_verts": 9.26, "K": 3,
         "queries": 100},
        # short tuples on a database of 300,000 (64 x 2 bands): hundreds of candidates a query
        {"name": "shortlist_dense", "kind": "shortlist", "shape": "scale", "polys": 300_000, "K": 128,
         "bands": 64, "queries": 4096, "m": 64},
        # a full query batch through the captured graph, plain form, refined to the top ten
        {"name": "search_batch", "kind": "search", "polys": 400_000, "K": 128, "bands": 32,
         "queries": 4096, "m": 19, "k": 10, "learned": False, "shortlist": 0},
        # one query through its graph, learned form: the smallest serving call
        {"name": "search_one", "kind": "search", "polys": 200_000, "K": 128, "bands": 64, "queries": 1,
         "m": 17, "k": 10, "learned": True, "shortlist": 32},
        # ground truth of a recall measurement: every box-overlapping pair refined exactly
        {"name": "truth_combined", "kind": "truth", "shape": "combined", "polys": 100_000, "queries": 96},
        # exact refinement of coastlines of up to 16,384 vertices against their candidates
        {"name": "refine_coastline", "kind": "refine", "polys": 2000, "max_verts": 16384, "queries": 64,
         "per_query": 8},
        # scoring a batch's shortlists (4,096 x 64 pairs) and keeping the best 32 of each
        {"name": "score_batch", "kind": "score", "queries": 4096, "shortlist": 64, "m": 32},
        # one minibatch of reranker training (the training loop's batch of 4,096 pairs)
        {"name": "train_batch", "kind": "gradients", "rows": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["sign", "sign", "sign", "ingest", "hashmap", "shortlist", "search", "search",
                       "truth", "refine", "score", "gradients"])
    if kind == "sign":
        shape = rng.choice(["small", "scale", "combined", "coastline"])
        if shape == "small":
            return {"kind": kind, "shape": shape, "polys": _log_int(rng, 100, 20_000), "max_verts": 0,
                    "K": rng.choice([7, 32, 40, 64, 96]), "index": rng.random() < 0.5}
        if shape == "coastline":
            return {"kind": kind, "shape": shape, "polys": _log_int(rng, 100, 8000),
                    "max_verts": _log_int(rng, 1024, 65536), "K": rng.choice([64, 96, 128, 256]),
                    "index": True}
        return {"kind": kind, "shape": shape, "polys": _log_int(rng, 1000, 300_000), "max_verts": 0,
                "K": rng.choice([32, 64, 96, 128]), "index": True}
    if kind == "ingest":
        return {"kind": kind, "shape": rng.choice(["scale", "combined"]),
                "polys": _log_int(rng, 10_000, 400_000), "K": 128, "bands": rng.choice([8, 16, 32]),
                "queries": rng.randint(64, 512)}
    if kind == "hashmap":
        return {"kind": kind, "polys": _log_int(rng, 5_000, 149_000), "mean_verts": rng.choice([9.26, 12.0]),
                "K": rng.randint(1, 5), "queries": rng.randint(20, 100)}
    if kind == "shortlist":
        return {"kind": kind, "shape": rng.choice(["scale", "combined"]),
                "polys": _log_int(rng, 20_000, 300_000), "K": 128, "bands": rng.choice([8, 16, 32, 64]),
                "queries": _log_int(rng, 64, 4096), "m": rng.randint(8, 64)}
    if kind == "search":
        learned = rng.random() < 0.5
        return {"kind": kind, "polys": _log_int(rng, 20_000, 300_000), "K": 128,
                "bands": rng.choice([16, 32, 64]), "queries": _log_int(rng, 1, 4096),
                "m": rng.randint(10, 24), "k": 10, "learned": learned, "shortlist": 32 if learned else 0}
    if kind == "truth":
        return {"kind": kind, "shape": rng.choice(["scale", "combined"]),
                "polys": _log_int(rng, 10_000, 100_000), "queries": rng.randint(16, 96)}
    if kind == "refine":
        return {"kind": kind, "polys": rng.randint(500, 2000), "max_verts": _log_int(rng, 512, 12_000),
                "queries": rng.randint(16, 64), "per_query": rng.randint(4, 8)}
    if kind == "score":
        return {"kind": kind, "queries": _log_int(rng, 16, 4096), "shortlist": rng.randint(24, 64),
                "m": rng.randint(8, 24)}
    return {"kind": kind, "rows": _log_int(rng, 512, 65_536)}


# ---------------------------------------------------------------------------
# what a program keeps between calls
# ---------------------------------------------------------------------------
_contexts = {}


def _context(params):
    """One context per signature length, its stream index built once, production kernels."""
    ctx = _contexts.get(params.K)
    if ctx is None:
        ctx = _contexts[params.K] = B.Context(0)
        B.sign_count_work(ctx, False)
    if params.flags & B.FLAG_STREAM_INDEX:
        B.stream_index_build(ctx, params)
    return ctx


def _params(K, bands, index=True):
    return B.make_params(K, bands, T24, SEED, LSH_SEED, B.FLAG_STREAM_INDEX if index else 0)


def _polygons(shape, n, seed, max_verts=0):
    s = dict(_SHAPES[shape])
    if max_verts:
        s["n_range"] = (s["n_range"][0], max_verts)
    return synth.star_polygons(n, 1000 + seed, **s)


def _device(ps):
    return torch.from_numpy(ps.xy).cuda(), torch.from_numpy(ps.offsets).cuda()


# mean share of a database that a query meets: in its buckets, by family and bands (K = 128);
# in the single hashmap of a centred set, by K; by bounding box
_IN_BUCKETS = {"combined": {8: 3e-5, 16: 4e-5, 32: 2.6e-4, 64: 1.7e-3},
               "scale": {8: 3e-5, 16: 8e-5, 32: 6e-4, 64: 3.2e-3}}
_IN_HASHMAP = {1: 0.55, 2: 0.25, 3: 0.12, 4: 0.09, 5: 0.07}
_IN_BOX = {"combined": 0.0066, "scale": 0.017}


def _share(case):
    if case["kind"] == "hashmap":
        return _IN_HASHMAP[case["K"]]
    if case["kind"] == "truth":
        return _IN_BOX[case["shape"]]
    return _IN_BUCKETS[case.get("shape", "combined")][case["bands"]]


def _capacity(case):
    """Size of a program's own result arrays for the candidates of one pass."""
    return int(case["polys"] * _share(case) * (1.5 * case["queries"] + 16)) + 24 * case["queries"] + 4096


def _result(case, dtype):
    return torch.zeros(_capacity(case), dtype=dtype, device="cuda")


def _store(buf, values):
    """Keep a pass's values in the program's array (whose tail stays zero)."""
    buf[:values.numel()].copy_(values)
    return buf


def _upload(ctx, ps):
    xy, off = _device(ps)
    return B.poly_upload(ctx, xy, off)


def _truth_inputs(case, seed):
    db = _polygons(case["shape"], case["polys"], seed)
    return db, synth.perturbed_queries(db, case["queries"], 5000 + seed)


def _boxes(ps):
    """Bounding boxes clipped to the domain (x0, y0, x1, y1)."""
    lo = np.minimum.reduceat(ps.xy, ps.offsets[:-1], axis=0)
    hi = np.maximum.reduceat(ps.xy, ps.offsets[:-1], axis=0)
    return np.concatenate([np.clip(lo, 0, synth.DOMAIN), np.clip(hi, 0, synth.DOMAIN)], axis=1)


def _overlapping(a, boxes):
    return np.flatnonzero((a[0] < boxes[:, 2]) & (boxes[:, 0] < a[2]) & (a[1] < boxes[:, 3]) &
                          (boxes[:, 1] < a[3]))


def _refine_inputs(case, seed):
    """Queries, database and pairs: each query with its source and the overlapping polygons
    nearest to it in area (what a shortlist of similar polygons holds)."""
    db = _polygons("coastline", case["polys"], seed, case["max_verts"])
    qs = synth.perturbed_queries(db, case["queries"], 5000 + seed)
    boxes, qboxes = _boxes(db), _boxes(qs)
    size = np.log(np.maximum(db.rbar, 1.0))
    qid, pid = [], []
    for q in range(qs.n):
        apart = np.ones(db.n, np.int64)  # (where too few overlap, the nearest in area follow)
        apart[_overlapping(qboxes[q], boxes)] = 0
        near = np.lexsort((np.abs(size - math.log(max(qs.rbar[q], 1.0))), apart))
        near = near[near != qs.source[q]][:case["per_query"] - 1]
        ids = np.concatenate([[qs.source[q]], near])
        qid.append(np.full(len(ids), q))
        pid.append(ids)
    return qs, db, np.concatenate(qid).astype(np.int32), np.concatenate(pid).astype(np.int32)


def _features(rows, seed):
    """Feature rows (bf16 bits [rows, 48]) and labels distributed as those of (query, candidate)
    pairs: agreement a, group bits with probability ~a^4, log areas and vertex counts, order
    counts, box bound; the label is a noisy a."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def rand(*shape):
        return torch.rand(*shape, generator=g, device="cuda")

    a = rand(rows) ** 2
    x = torch.zeros(rows, 48, device="cuda")
    x[:, :32] = (rand(rows, 32) < (a ** 4)[:, None]).float()
    x[:, 32] = torch.round(a * 128) / 128
    area = 0.45 + 0.35 * rand(rows)
    verts = 0.2 + 0.4 * rand(rows)
    x[:, 33], x[:, 34] = area, area + 0.02 * (rand(rows) - 0.5)
    x[:, 35], x[:, 36] = verts, verts + 0.05 * (rand(rows) - 0.5)
    lt = (1 - x[:, 32]) * (0.3 + 0.4 * rand(rows))
    x[:, 37], x[:, 38] = lt, 1 - x[:, 32] - lt
    x[:, 39] = torch.clamp(a + (1 - a) * rand(rows), max=1.0)
    label = torch.clamp(a + 0.05 * (rand(rows) - 0.5), 0.0, 1.0)
    return x.to(torch.bfloat16).view(torch.int16).contiguous(), label


def prepare(case, seed):
    kind = case["kind"]
    if kind == "sign":
        P = _params(case["K"], 1, case["index"])
        ctx = _context(P)
        polys = _upload(ctx, _polygons(case["shape"], case["polys"], seed, case["max_verts"]))
        return {"kind": kind, "ctx": ctx, "P": P, "polys": polys}
    if kind == "ingest":
        P = _params(case["K"], case["bands"])
        ctx = _context(P)
        db = _polygons(case["shape"], case["polys"], seed)
        xy, off = _device(db)
        polys = B.poly_upload(ctx, xy, off)
        qp = _upload(ctx, synth.perturbed_queries(db, case["queries"], 5000 + seed))
        hashes = B.minhash_sign(ctx, polys, P)
        return {"kind": kind, "ctx": ctx, "P": P, "xy": xy, "off": off, "polys": polys, "hashes": hashes,
                "qh": B.minhash_sign(ctx, qp, P), "index": B.lsh_build(ctx, hashes, P),
                "cand": _result(case, torch.int32)}
    if kind == "hashmap":
        P = _params(case["K"], 1)
        ctx = _context(P)
        db = synth.paper_shaped(case["polys"], case["mean_verts"], 1000 + seed)
        h = B.minhash_sign(ctx, _upload(ctx, db), P)
        qh = B.minhash_sign(ctx, _upload(ctx, synth.paper_queries(db, case["queries"], 5000 + seed)), P)
        return {"kind": kind, "ctx": ctx, "index": B.lsh_build(ctx, h, P), "qh": qh,
                "cand": _result(case, torch.int32)}
    if kind == "shortlist":
        P = _params(case["K"], case["bands"])
        ctx = _context(P)
        db = _polygons(case["shape"], case["polys"], seed)
        h = B.minhash_sign(ctx, _upload(ctx, db), P)
        qh = B.minhash_sign(ctx, _upload(ctx, synth.perturbed_queries(db, case["queries"], 5000 + seed)), P)
        return {"kind": kind, "ctx": ctx, "P": P, "h": h, "qh": qh, "index": B.lsh_build(ctx, h, P),
                "m": case["m"], "cand": _result(case, torch.int32), "count": _result(case, torch.int16),
                "mask": _result(case, torch.int32)}
    if kind == "search":
        P = _params(case["K"], case["bands"])
        ctx = _context(P)
        db = _polygons("combined", case["polys"], seed)
        dbp = _upload(ctx, db)
        index = B.lsh_build(ctx, B.minhash_sign(ctx, dbp, P), P)
        qs = synth.perturbed_queries(db, case["queries"], 5000 + seed)
        qxy, qoff = _device(qs)
        rr = B.Reranker(ctx, seed=seed) if case["learned"] else None
        g = B.QueryGraph(ctx, index, qs.n, qs.n_vertices, _capacity(case), case["m"], db=dbp, k=case["k"],
                         rerank=rr, shortlist=case["shortlist"])
        g.cand.zero_()
        g.count.zero_()
        return {"kind": kind, "graph": g, "xy": qxy, "off": qoff}
    if kind == "truth":
        ctx = _context(_params(128, 16))
        db, qs = _truth_inputs(case, seed)
        return {"kind": kind, "ctx": ctx, "db": _upload(ctx, db), "q": _upload(ctx, qs),
                "cand": _result(case, torch.int32), "j": _result(case, torch.float64)}
    if kind == "refine":
        ctx = _context(_params(128, 16))
        qs, db, qid, pid = _refine_inputs(case, seed)
        return {"kind": kind, "ctx": ctx, "db": _upload(ctx, db), "q": _upload(ctx, qs),
                "qid": torch.from_numpy(qid).cuda(), "pid": torch.from_numpy(pid).cuda()}
    ctx = _context(_params(128, 16))
    rr = B.Reranker(ctx, weights=B.init_rerank_params(seed))
    if kind == "score":
        Q, S = case["queries"], case["shortlist"]
        feat, _ = _features(Q * S, seed)
        g = torch.Generator(device="cuda")
        g.manual_seed(seed + 1)
        step = torch.randint(1, 5000, (Q, S), generator=g, device="cuda", dtype=torch.int32)
        cand = torch.cumsum(step, dim=1, dtype=torch.int32).reshape(-1).contiguous()
        row_ptr = torch.arange(Q + 1, device="cuda", dtype=torch.int64) * S
        return {"kind": kind, "ctx": ctx, "rr": rr, "feat": feat, "cand": cand, "row_ptr": row_ptr,
                "m": case["m"]}
    feat, label = _features(case["rows"], seed)
    return {"kind": kind, "rr": rr, "feat": feat, "label": label}


def _kept(graph, view):
    """A view of a graph's buffer that keeps the graph (its memory's owner) alive."""
    out = view[:]
    out.graph = graph
    return out


def run(s):
    kind = s["kind"]
    if kind == "sign":
        return {"hashes": B.minhash_sign(s["ctx"], s["polys"], s["P"])}
    if kind == "ingest":
        B.poly_reload(s["polys"], s["xy"], s["off"])
        bbox, area2 = s["polys"].prep()
        hashes = B.minhash_sign(s["ctx"], s["polys"], s["P"], out=s["hashes"])
        B.lsh_rebuild(s["ctx"], s["index"], hashes)
        row_ptr, cand = B.lsh_query(s["ctx"], s["index"], s["qh"])
        return {"bbox": bbox, "area2": area2, "hashes": hashes, "row_ptr": row_ptr,
                "cand": _store(s["cand"], cand)}
    if kind == "hashmap":
        row_ptr, cand = B.lsh_query(s["ctx"], s["index"], s["qh"])
        return {"row_ptr": row_ptr, "cand": _store(s["cand"], cand)}
    if kind == "shortlist":
        row_ptr, cand = B.lsh_query(s["ctx"], s["index"], s["qh"])
        count, mask = B.jaccard_estimate(s["ctx"], s["qh"], s["h"], row_ptr, cand, s["P"])
        ids, n = B.topm(s["ctx"], row_ptr, cand, count, s["m"])
        return {"row_ptr": row_ptr, "cand": _store(s["cand"], cand), "count": _store(s["count"], count),
                "mask": _store(s["mask"], mask), "ids": ids, "n": n}
    if kind == "search":
        g = s["graph"]
        g.run(s["xy"], s["off"])
        views = {"hashes": g.hashes, "row_ptr": g.row_ptr, "cand": g.cand, "count": g.count, "top_ids": g.top_ids,
                 "top_n": g.top_n, "ref_ids": g.ref_ids, "ref_j": g.ref_j}
        return {name: _kept(g, v) for name, v in views.items()}
    if kind == "truth":
        row_ptr, cand = B.bbox_join(s["ctx"], s["q"], s["db"])
        qid = torch.repeat_interleave(torch.arange(s["q"].n, device="cuda", dtype=torch.int32),
                                      row_ptr[1:] - row_ptr[:-1])
        j = B.pair_jaccard(s["ctx"], s["q"], s["db"], qid, cand)
        return {"row_ptr": row_ptr, "cand": _store(s["cand"], cand), "j": _store(s["j"], j)}
    if kind == "refine":
        return {"j": B.pair_jaccard(s["ctx"], s["q"], s["db"], s["qid"], s["pid"])}
    if kind == "score":
        score = s["rr"].forward(s["feat"])
        ids, n = B.topm(s["ctx"], s["row_ptr"], s["cand"], None, s["m"], score=score)
        return {"score": score, "ids": ids, "n": n}
    grads, loss = s["rr"].gradients(s["feat"], s["label"])
    return {"grads": grads, "loss": loss}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _mean_verts(shape, max_verts=0):
    (lo, hi), dist = _SHAPES[shape]["n_range"], _SHAPES[shape]["n_dist"]
    hi = max_verts or hi
    return 0.5 * (lo + hi) if dist == "uniform" else (hi - lo) / math.log(hi / lo)


def work(case):
    kind = case["kind"]
    if kind == "sign":
        n = case["polys"]
        verts = n * _mean_verts(case["shape"], case["max_verts"])
        return {"bytes": 8 * verts + 8 * n + 4 * n * case["K"], "flops": 0}
    if kind == "ingest":
        # vertices and offsets in and kept, boxes and areas out, hashes out and kept, one
        # (key, id) entry per polygon and band
        n = case["polys"]
        verts = n * _mean_verts(case["shape"])
        return {"bytes": 16 * verts + n * (16 + 24 + 8 * case["K"] + 8 * case["bands"]), "flops": 0}
    if kind == "hashmap":  # an id in and out per candidate
        return {"bytes": 8 * case["queries"] * case["polys"] * _share(case), "flops": 0}
    if kind == "shortlist":  # each candidate's hashes, id, count and band bits, the queries and lists
        pairs = case["queries"] * case["polys"] * _share(case)
        return {"bytes": pairs * (4 * case["K"] + 14) + case["queries"] * 4 * (case["K"] + case["m"]), "flops": 0}
    if kind == "search":  # the queries' vertices, the candidates' hashes, the refined rings, the lists
        verts, Q = _mean_verts("combined"), case["queries"]
        pairs = Q * case["polys"] * _share(case)
        return {"bytes": 8 * verts * Q * (1 + case["m"]) + pairs * (4 * case["K"] + 10)
                + Q * (4 * case["K"] + 4 * case["m"] + 12 * case["k"]), "flops": 0}
    if kind == "truth":  # the boxes once, and each pair's rings, id and result
        pairs = case["queries"] * case["polys"] * _share(case)
        return {"bytes": 16 * case["polys"] + pairs * (16 + 16 * _mean_verts(case["shape"])), "flops": 0}
    if kind == "refine":
        pairs = case["queries"] * case["per_query"]
        return {"bytes": pairs * (16 * _mean_verts("coastline", case["max_verts"]) + 16), "flops": 0}
    mlp = 2 * (40 * 64 + 64 * 64 + 64)
    if kind == "score":
        rows = case["queries"] * case["shortlist"]
        return {"bytes": rows * (96 + 4 + 4) + case["queries"] * 4 * (case["m"] + 1), "flops": rows * mlp}
    return {"bytes": case["rows"] * 100 + 8 * B.RERANK_PARAMS, "flops": 3 * case["rows"] * mlp}


# ---------------------------------------------------------------------------
# the same values in 64 bits
# ---------------------------------------------------------------------------
def _pair_jaccard64(qs, db, qid, pid, chunk=1 << 23):
    """Jaccard of every (query, database) pair: a simple polygon's indicator is the signed sum of
    its edges' trapezoids down to a base line, so area(A n B) is the signed sum over edge pairs of
    the integral of the smaller of the two edges' heights over their common x-range."""
    dev = "cuda"

    def ring(ps):
        xy = torch.from_numpy(ps.xy).to(dev, torch.float64)
        off = torch.from_numpy(ps.offsets).to(dev)
        nxt = torch.arange(len(xy), device=dev) + 1
        nxt[off[1:] - 1] = off[:-1]
        nx = xy[nxt]
        cr = xy[:, 0] * nx[:, 1] - nx[:, 0] * xy[:, 1]
        c = torch.cat([torch.zeros(1, device=dev, dtype=torch.float64), torch.cumsum(cr, 0)])
        return xy, nx, off, 0.5 * (c[off[1:]] - c[off[:-1]])

    ax, an, aoff, aarea = ring(qs)
    bx, bn, boff, barea = ring(db)
    qid = torch.as_tensor(qid, device=dev).long()
    pid = torch.as_tensor(pid, device=dev).long()
    na, nb = (aoff[1:] - aoff[:-1])[qid], (boff[1:] - boff[:-1])[pid]
    start = torch.cat([torch.zeros(1, device=dev, dtype=torch.int64), torch.cumsum(na * nb, 0)])
    inter = torch.zeros(len(qid), device=dev, dtype=torch.float64)
    total = int(start[-1])
    for s in range(0, total, chunk):
        t = torch.arange(s, min(s + chunk, total), device=dev)
        e = torch.searchsorted(start, t, right=True) - 1
        r = t - start[e]
        i, j = aoff[qid[e]] + r // nb[e], boff[pid[e]] + r % nb[e]
        p, q, u, v = ax[i], an[i], bx[j], bn[j]
        base = bx[boff[pid[e]]]  # heights and abscissae relative to the database polygon's first vertex
        p, q, u, v = p - base, q - base, u - base, v - base
        sgn = torch.sign(q[:, 0] - p[:, 0]) * torch.sign(v[:, 0] - u[:, 0])
        l = torch.maximum(torch.minimum(p[:, 0], q[:, 0]), torch.minimum(u[:, 0], v[:, 0]))
        h = torch.minimum(torch.maximum(p[:, 0], q[:, 0]), torch.maximum(u[:, 0], v[:, 0]))
        ok = (sgn != 0) & (h > l)
        e, p, q, u, v, l, h, sgn = e[ok], p[ok], q[ok], u[ok], v[ok], l[ok], h[ok], sgn[ok]
        ma, mb = (q[:, 1] - p[:, 1]) / (q[:, 0] - p[:, 0]), (v[:, 1] - u[:, 1]) / (v[:, 0] - u[:, 0])
        al, ah = p[:, 1] + ma * (l - p[:, 0]), p[:, 1] + ma * (h - p[:, 0])
        bl, bh = u[:, 1] + mb * (l - u[:, 0]), u[:, 1] + mb * (h - u[:, 0])
        dl, dh = al - bl, ah - bh
        val = 0.5 * (torch.minimum(al, bl) + torch.minimum(ah, bh)) * (h - l)
        cross = dl * dh < 0  # the heights cross inside: the smaller one has a kink there
        dl, dh = dl.abs(), dh.abs()
        val = val + torch.where(cross, 0.5 * (h - l) * dl * dh / (dl + dh).clamp_min(1e-300), torch.zeros_like(val))
        inter.index_add_(0, e, sgn * val)
    sign = torch.sign(aarea[qid]) * torch.sign(barea[pid])
    inter = inter * sign
    uni = aarea[qid].abs() + barea[pid].abs() - inter
    return torch.where(uni > 0, (inter / uni).clamp(0.0, 1.0), torch.zeros_like(uni))


def _unpack(seed):
    """The network's weights in 64 bits (packed layout of the header: w1, b1, w2, b2, w3, b3)."""
    w = torch.from_numpy(np.array(B.init_rerank_params(seed), np.float64)).cuda()
    return [t.reshape(shape) for t, shape in zip(torch.split(w, [64 * 40, 64, 64 * 64, 64, 64, 1]),
                                                 [(64, 40), (64,), (64, 64), (64,), (64,), (1,)])]


def _predict(weights, feat):
    w1, b1, w2, b2, w3, b3 = weights
    x = feat.view(torch.bfloat16)[:, :40].to(torch.float64)
    h = torch.relu(torch.relu(x @ w1.T + b1) @ w2.T + b2)
    return torch.sigmoid(h @ w3 + b3)


def exact(case, seed):
    kind = case["kind"]
    if kind == "truth":
        db, qs = _truth_inputs(case, seed)
        boxes, qboxes = _boxes(db), _boxes(qs)
        rows = [_overlapping(qboxes[q], boxes) for q in range(qs.n)]
        qid = np.repeat(np.arange(qs.n), [len(r) for r in rows])
        j = _pair_jaccard64(qs, db, qid, np.concatenate(rows))
        return {"row_ptr": None, "cand": None, "j": _store(_result(case, torch.float64), j)}
    if kind == "refine":
        qs, db, qid, pid = _refine_inputs(case, seed)
        return {"j": _pair_jaccard64(qs, db, qid, pid)}
    if kind == "score":
        feat, _ = _features(case["queries"] * case["shortlist"], seed)
        return {"score": _predict(_unpack(seed), feat), "ids": None, "n": None}
    if kind == "gradients":
        feat, label = _features(case["rows"], seed)
        weights = [w.clone().requires_grad_(True) for w in _unpack(seed)]
        loss = ((_predict(weights, feat) - label.to(torch.float64)) ** 2).mean()
        grads = torch.autograd.grad(loss, weights)
        return {"grads": torch.cat([g.reshape(-1) for g in grads]), "loss": loss.detach().reshape(1)}
    # hashes, candidates, counts and lists are whole numbers; the searches' Jaccards belong to
    # pairs that only the hashes pick
    return None
