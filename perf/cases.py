"""Performance cases of the matching library: what a user of it has it do, over the range of sizes it is used at.

Each case is one call, or one chain of calls, of the public Python entry points. ``prepare`` makes what the caller has
in hand before the call (inputs, a built index, an installed second inverted file), ``run`` is the call itself,
``work`` the bytes and operations it cannot do without, and ``exact`` the same outputs in 64 bits in plain torch.

Features follow the recipe of the repository's workloads: a view is ReLU(class centre + 0.3 noise), L2-normalised, so
views of a class form a cloud and lists are uneven. Vocabularies are two Lloyd steps over a sample of the database
views. Neighbour rows (for second inverted files that are installed, not built) are members of a shape's own class
drawn with a per-shape popularity, so entries of the inverted file have uneven lengths too.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1604_01879_gb300 as gift

NOISE = 0.3


def listed():
    return [
        # A WM-SHREC07-sized database, FP32 store, ten queries and their re-rank: a call whose arithmetic takes
        # microseconds, so launches and latency are what a user sees.
        {"name": "small_f32_step", "kind": "query", "shapes": 200, "views": 64, "dim": 128, "classes": 20,
         "codewords": 64, "storage": "f32", "ma": 1, "rescore": 0, "queries": 10, "query_views": "64", "topk": 10,
         "k1": 10},
        # The serving loop's ordinary batch: a handful of requests of mixed view counts against an FP8 index with
        # query-side multiple assignment and FP32 rescore, re-ranked.
        {"name": "serving_fp8_step", "kind": "query", "shapes": 3200, "views": 64, "dim": 4096, "classes": 64,
         "codewords": 512, "storage": "fp8", "ma": 2, "rescore": 100, "queries": 4, "query_views": "12,20,64",
         "topk": 100, "k1": 50},
        # The large-database step: 256 queries per batch, FP8 store, MA = 2, rescore, re-rank.
        {"name": "batch_fp8_step", "kind": "query", "shapes": 20000, "views": 64, "dim": 4096, "classes": 400,
         "codewords": 4096, "storage": "fp8", "ma": 2, "rescore": 200, "queries": 256, "query_views": "64",
         "topk": 100, "k1": 50},
        # The ModelNet40-sized step: 1,000 queries against a BF16 store with two-part rescore rows, and the re-rank.
        {"name": "batch_bf16_step", "kind": "query", "shapes": 12000, "views": 64, "dim": 4096, "classes": 40,
         "codewords": 1024, "storage": "bf16", "ma": 1, "rescore": 200, "queries": 1000, "query_views": "64",
         "topk": 100, "k1": 50},
        # The plain path: Eq. 3 over all view pairs, which a user runs to check an index's recall.
        {"name": "exact_bf16", "kind": "exact", "shapes": 2000, "views": 64, "dim": 4096, "classes": 40,
         "codewords": 1024, "storage": "bf16", "ma": 1, "rescore": 200, "queries": 16, "query_views": "64",
         "topk": 100, "k1": 0},
        # Re-ranking alone over a 200,000-shape second inverted file (a shard re-ranks merged candidates this way).
        {"name": "rerank_200k", "kind": "rerank", "shapes": 200000, "classes": 400, "queries": 256, "cand": 100,
         "k1": 50, "topk": 100},
        # The paper's default re-rank: two similarity measures, co-augmentation, k2 = 4, alpha = 0.5.
        {"name": "two_measure_rerank", "kind": "aca", "shapes": 12000, "classes": 40, "queries": 1000, "cand": 100,
         "k1": 50, "k2": 4, "topk": 100},
        # Training the projection at full size: forward (scores and saved argmax) ...
        {"name": "match_forward_bf16", "kind": "forward", "queries": 256, "query_views": "64", "shapes": 4096,
         "views": 64, "din": 4096, "dout": 512, "dtype": "bf16", "classes": 40},
        # ... and backward (gradients of the projection and of both view sets).
        {"name": "match_backward_bf16", "kind": "backward", "queries": 256, "query_views": "64", "shapes": 4096,
         "views": 64, "din": 4096, "dout": 512, "dtype": "bf16", "classes": 40},
        # A small FP32 training step through autograd, ragged queries and an odd number of views.
        {"name": "train_step_f32", "kind": "step", "queries": 24, "query_views": "12,20,64", "shapes": 333, "views": 20,
         "din": 512, "dout": 128, "dtype": "f32", "classes": 20},
        # The off-line vocabulary.
        {"name": "kmeans_16k", "kind": "kmeans", "rows": 16384, "dim": 4096, "codewords": 1024, "iters": 10,
         "classes": 40},
        # The projection front end: 64 depth views of every mesh.
        {"name": "render_224", "kind": "render", "meshes": 64, "n_lat": 24, "n_lon": 48, "n_az": 8, "n_el": 8,
         "side": 224},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_query(rng, kind):
    storage = rng.choice(("f32", "bf16", "bf16", "fp8", "fp8")) if kind == "query" else rng.choice(("bf16", "fp8"))
    if storage == "f32":
        classes, dim = _log(rng, 5, 40), 16 * _log(rng, 4, 16)
        members, queries, views = _log(rng, 5, 25), _log(rng, 1, 64), rng.randint(8, 64)
    elif kind == "exact":
        classes, dim = _log(rng, 8, 40), 16 * _log(rng, 16, 256)
        members, queries, views = _log(rng, 10, 50), _log(rng, 1, 16), rng.choice((12, 20, 33, 64))
    else:
        classes, dim = _log(rng, 16, 200), 16 * _log(rng, 16, 256)
        members, queries, views = _log(rng, 8, 50), _log(rng, 1, 256), rng.choice((12, 20, 33, 64))
    shapes = classes * members
    topk = min(shapes, rng.choice((10, 50, 100)))
    return {"kind": kind, "shapes": shapes, "views": views, "dim": dim, "classes": classes,
            "codewords": min(4096, classes * rng.randint(2, 10)), "storage": storage,
            "ma": 1 if kind == "exact" else rng.choice((1, 2)),
            "rescore": 0 if storage == "f32" else min(shapes, topk * rng.randint(1, 3)), "queries": queries,
            "query_views": rng.choice(("64", "12,20,64", "20", "7,33")), "topk": topk,
            "k1": 0 if kind == "exact" else min(topk, members, rng.choice((5, 10, 50)))}


def draw(rng):
    """One more case of the listed ranges."""
    kind = rng.choice(("query", "query", "query", "exact", "rerank", "aca", "forward", "backward", "step", "kmeans",
                       "render"))
    if kind in ("query", "exact"):
        return _draw_query(rng, kind)
    if kind == "rerank":
        classes, members = _log(rng, 4, 400), _log(rng, 60, 500)
        k1 = rng.choice((10, 25, 50))
        return {"kind": kind, "shapes": classes * members, "classes": classes, "queries": _log(rng, 1, 256),
                "cand": rng.randint(k1, 59), "k1": k1, "topk": rng.choice((10, 37, 100))}
    if kind == "aca":
        classes, members = _log(rng, 4, 40), _log(rng, 60, 300)
        k1 = rng.choice((10, 25, 50))
        return {"kind": kind, "shapes": classes * members, "classes": classes, "queries": _log(rng, 1, 1000),
                "cand": rng.randint(k1, 59), "k1": k1, "k2": rng.randint(1, 4), "topk": rng.choice((10, 37, 100))}
    if kind in ("forward", "backward", "step"):
        return {"kind": kind, "queries": _log(rng, 4, 200), "query_views": rng.choice(("64", "12,20,64", "20", "7,33")),
                "shapes": _log(rng, 40, 3000), "views": rng.choice((12, 20, 33, 64, 64)), "din": 16 * _log(rng, 8, 256),
                "dout": 16 * _log(rng, 4, 32), "dtype": rng.choice(("f32", "bf16")), "classes": _log(rng, 5, 40)}
    if kind == "kmeans":
        return {"kind": kind, "rows": _log(rng, 1024, 16384), "dim": 16 * _log(rng, 8, 256),
                "codewords": _log(rng, 16, 1000), "iters": rng.randint(2, 8), "classes": _log(rng, 5, 40)}
    return {"kind": kind, "meshes": _log(rng, 1, 60), "n_lat": rng.randint(6, 24), "n_lon": rng.randint(8, 48),
            "n_az": rng.randint(1, 8), "n_el": rng.randint(1, 8), "side": _log(rng, 32, 224)}


# ---------------------------------------------------------------- inputs
def _gen(seed, stream=0):
    return torch.Generator(device="cuda").manual_seed(1_000_003 * int(seed) + int(stream))


def _views(n, per, dim, centres, gen):
    """[n * per, dim] L2-normalised views; shape s has class s mod the number of centres."""
    out = torch.empty((n * per, dim), device="cuda")
    step = max(1, (1 << 28) // (per * dim))
    for s in range(0, n, step):
        m = min(step, n - s)
        cls = torch.arange(s, s + m, device="cuda") % centres.shape[0]
        v = torch.randn((m, per, dim), generator=gen, device="cuda").mul_(NOISE).add_(centres[cls][:, None]).relu_()
        v.div_(v.norm(dim=2, keepdim=True).clamp_min_(1e-20))
        out[s * per:(s + m) * per] = v.view(m * per, dim)
    return out


def _query_views(case, centres, seed):
    """Views of every query (flat) and the int32 offsets; the case's view counts take turns."""
    choices = [int(x) for x in case["query_views"].split(",")]
    counts = np.resize(choices, case["queries"])
    offs = np.zeros(case["queries"] + 1, np.int32)
    offs[1:] = np.cumsum(counts)
    full = _views(case["queries"], max(choices), centres.shape[1], centres, _gen(seed, 2))
    keep = torch.from_numpy((np.arange(max(choices))[None, :] < counts[:, None]).reshape(-1)).cuda()
    return full[keep].contiguous(), offs


def _codebook(db, k, gen):
    """Two Lloyd steps over a sample of the views, from k of them."""
    n = db.shape[0]
    x = db[torch.randperm(n, generator=gen, device="cuda")[:max(k, min(n, 16384))]]
    if x.shape[0] < k:
        x = x[torch.arange(k, device="cuda") % x.shape[0]]
    cb = x[:k].clone()
    for _ in range(2):
        near = (x @ cb.T - 0.5 * (cb * cb).sum(1)).argmax(1)
        pick = torch.nn.functional.one_hot(near, k).float().T.contiguous()
        size = pick.sum(1, keepdim=True)
        cb = torch.where(size > 0, (pick @ x) / size.clamp_min(1.0), cb)
    return cb.contiguous()


def _query_inputs(case, seed):
    centres = torch.randn((case["classes"], case["dim"]), generator=_gen(seed), device="cuda")
    db = _views(case["shapes"], case["views"], case["dim"], centres, _gen(seed, 1))
    q, offs = _query_views(case, centres, seed)
    return db, q, offs, _codebook(db, case["codewords"], _gen(seed, 3))


def _neighbours(shapes, classes, k, gen, first_self=True, rows=None):
    """Ranked neighbour rows (ids int32, scores float32) [rows, k]: distinct members of the row's class, scores
    descending; row r of a database starts with r itself."""
    members = shapes // classes
    r = torch.arange(shapes if rows is None else rows, device="cuda")
    cls = r % classes
    pop = 0.5 * torch.rand((classes, members), generator=gen, device="cuda")
    ids = torch.empty((r.numel(), k), dtype=torch.int32, device="cuda")
    for s in range(0, r.numel(), 16384):
        c = cls[s:s + 16384]
        w = torch.rand((c.numel(), members), generator=gen, device="cuda") + pop[c]
        if first_self:
            w.scatter_(1, (r[s:s + 16384] // classes)[:, None], 2.0)
        ids[s:s + 16384] = (w.topk(k, dim=1).indices * classes + c[:, None]).int()
    sc = (0.75 + 0.2 * torch.rand((r.numel(), k), generator=gen, device="cuda")).sort(1, descending=True).values
    if first_self:
        sc[:, 0] = 1.0
    return ids, sc.contiguous()


def _match_inputs(case, seed):
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    centres = torch.randn((case["classes"], case["din"]), generator=_gen(seed), device="cuda")
    p = _views(case["shapes"], case["views"], case["din"], centres, _gen(seed, 1))
    p = p.to(dt).view(case["shapes"], case["views"], case["din"])
    q, offs = _query_views(case, centres, seed)
    w = torch.randn((case["dout"], case["din"]), generator=_gen(seed, 4), device="cuda") / math.sqrt(case["dout"])
    g = torch.randn((case["queries"], case["shapes"]), generator=_gen(seed, 5), device="cuda")
    return q.to(dt), offs, p, w.to(dt), g


def _unit(x):
    return x / x.norm(dim=-1, keepdim=True).clamp_min(1e-300 if x.dtype == torch.float64 else 1e-30)


def _argmax(q, p, w, real):
    """The best database view of every (query view, shape) under the projection, evaluated in type `real`: (cosines,
    int16 indices)."""
    shapes, views, din = p.shape
    u = _unit(q.to(real) @ w.to(real).T)
    best = torch.empty((q.shape[0], shapes), dtype=real, device="cuda")
    arg = torch.empty((q.shape[0], shapes), dtype=torch.int16, device="cuda")
    step = max(1, (1 << 28) // (q.shape[0] * views))
    for s in range(0, shapes, step):
        v = _unit(p[s:s + step].reshape(-1, din).to(real) @ w.to(real).T)
        m = (u @ v.T).view(q.shape[0], -1, views).max(2)
        best[:, s:s + step], arg[:, s:s + step] = m.values, m.indices.short()
    return best, arg


def _mesh_inputs(case, seed):
    """Closed star-shaped surfaces on a latitude-longitude grid, bumped, stretched and shifted; the counts of vertices
    and triangles are those of the grid."""
    g = np.random.default_rng(int(seed))
    m, la, lo = case["meshes"], case["n_lat"], case["n_lon"]
    th = np.pi * np.arange(1, la) / la
    ph = 2 * np.pi * np.arange(lo) / lo
    t, f = (a.reshape(1, -1) for a in np.meshgrid(th, ph, indexing="ij"))
    r = np.ones((m, t.shape[1]))
    for _ in range(5):
        amp, a, b = g.uniform(0.05, 0.3, (m, 1)), g.integers(1, 5, (m, 1)), g.integers(1, 4, (m, 1))
        r += amp * np.cos(a * f + g.uniform(0, 6.28, (m, 1))) * np.sin(b * t + g.uniform(0, 6.28, (m, 1)))
    r = np.maximum(r, 0.2)
    ring = np.stack([r * np.sin(t) * np.cos(f), r * np.sin(t) * np.sin(f), r * np.cos(t)], -1)
    pole = np.broadcast_to(np.array([[[0.0, 0.0, 1.0]]]), (m, 1, 3))
    v = np.concatenate([pole, ring, -pole], 1) * g.uniform(0.6, 1.6, (m, 1, 3)) + g.uniform(-3, 3, (m, 1, 3))
    i, j = (a.reshape(-1) for a in np.meshgrid(np.arange(la - 2), np.arange(lo), indexing="ij"))
    at = lambda y, x: 1 + y * lo + x % lo  # noqa: E731
    k, last = np.arange(lo), v.shape[1] - 1
    tri = np.concatenate([
        np.stack([0 * k, at(0, k), at(0, k + 1)], 1), np.stack([0 * k + last, at(la - 2, k + 1), at(la - 2, k)], 1),
        np.stack([at(i, j), at(i + 1, j), at(i, j + 1)], 1), np.stack([at(i, j + 1), at(i + 1, j), at(i + 1, j + 1)], 1)])
    verts = torch.from_numpy(v.reshape(-1, 3).astype(np.float32)).cuda()
    tris = torch.from_numpy(np.tile(tri, (m, 1)).astype(np.int32)).cuda()
    return verts, tris, np.arange(m + 1) * v.shape[1], np.arange(m + 1) * len(tri)


def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("query", "exact"):
        db, s["q"], s["offs"], cb = _query_inputs(case, seed)
        s["index"] = gift.Index(db, cb, case["shapes"], case["views"], case["codewords"], storage=case["storage"],
                                query_ma=case["ma"], rescore_r=case["rescore"], keep_exact=kind == "exact")
        if case["k1"]:
            ids, sc = _neighbours(case["shapes"], case["classes"], case["k1"], _gen(seed, 6))
            s["index"].set_sif(ids, sc, case["shapes"], case["k1"])
    elif kind == "rerank":
        # a small shard that holds the replicated second inverted file of the whole database
        x = torch.rand((64, 16), generator=_gen(seed), device="cuda")
        s["index"] = gift.Index(x, x[:4].contiguous(), 64, 1, 4, keep_exact=False)
        ids, sc = _neighbours(case["shapes"], case["classes"], case["k1"], _gen(seed, 6))
        s["index"].set_sif(ids, sc, case["shapes"], case["k1"])
        s["cand"] = _neighbours(case["shapes"], case["classes"], case["cand"], _gen(seed, 7), False, case["queries"])
    elif kind == "aca":
        s["cand"] = []
        s["measures"] = []
        for m in range(2):
            x = torch.rand((case["shapes"], 16), generator=_gen(seed, 10 * m), device="cuda")
            ix = gift.Index(x, x[:4].contiguous(), case["shapes"], 1, 4, keep_exact=False)
            ids, sc = _neighbours(case["shapes"], case["classes"], case["k1"], _gen(seed, 10 * m + 1))
            ix.set_sif(ids, sc, case["shapes"], case["k1"])
            s["measures"].append(ix)
            s["cand"].append(_neighbours(case["shapes"], case["classes"], case["cand"], _gen(seed, 10 * m + 2), False,
                                         case["queries"]))
        s["aca"] = gift.Aca(s["measures"][0], s["measures"][1], k2=case["k2"], alpha=0.5, mode="co")
    elif kind in ("forward", "backward", "step"):
        s["q"], s["offs"], s["p"], s["w"], s["g"] = _match_inputs(case, seed)
        if kind == "backward":
            s["arg"] = _argmax(s["q"], s["p"], s["w"], torch.float32)[1]
        if kind == "step":
            for k in ("q", "p", "w"):
                s[k].requires_grad_(True)
    elif kind == "kmeans":
        centres = torch.randn((case["classes"], case["dim"]), generator=_gen(seed), device="cuda")
        s["x"] = _views(case["rows"], 1, case["dim"], centres, _gen(seed, 1))
        s["init"] = np.sort(np.random.default_rng(int(seed)).choice(case["rows"], case["codewords"], replace=False))
    else:
        s["mesh"] = _mesh_inputs(case, seed)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind in ("query", "exact"):
        ids, sc = s["index"].query(s["q"], s["offs"], mode="fif" if kind == "query" else "exact", topk=case["topk"])
        if not case["k1"]:
            return {"ids": ids, "scores": sc}
        ids2, sp = s["index"].rerank(ids, sc, k1=case["k1"], topk=case["topk"])
        return {"ids": ids, "scores": sc, "rerank_ids": ids2, "rerank_scores": sp}
    if kind == "rerank":
        ids, sp = s["index"].rerank(s["cand"][0], s["cand"][1], k1=case["k1"], topk=case["topk"])
        return {"ids": ids, "scores": sp}
    if kind == "aca":
        ids, sp = s["aca"].rerank(s["cand"][0], s["cand"][1], topk=case["topk"])
        return {"ids": ids, "scores": sp}
    if kind == "forward":
        score, arg = gift.match_forward(s["q"], s["offs"], s["p"], s["w"])
        return {"scores": score, "argmax": arg}
    if kind == "backward":
        dw, dq, dp = gift.match_backward(s["q"], s["offs"], s["p"], s["w"], s["g"], s["arg"])
        return {"dw": dw, "dq": dq, "dp": dp}
    if kind == "step":
        score = gift.GiftMatch.apply(s["q"], s["offs"], s["p"], s["w"])
        dq, dp, dw = torch.autograd.grad(score, (s["q"], s["p"], s["w"]), s["g"])
        return {"scores": score, "dw": dw, "dq": dq, "dp": dp}
    if kind == "kmeans":
        return gift.kmeans(s["x"], s["init"], case["iters"])
    return gift.render_views(*s["mesh"], n_az=case["n_az"], n_el=case["n_el"], H=case["side"], W=case["side"])


# ---------------------------------------------------------------- work
def _query_rows(case):
    return int(np.resize([int(x) for x in case["query_views"].split(",")], case["queries"]).sum())


def work(case):
    """Bytes (inputs once, outputs once) and multiply-adds x 2 of one pass."""
    kind = case["kind"]
    if kind in ("query", "exact"):
        nv, d, rows = _query_rows(case), case["dim"], case["shapes"] * case["views"]
        out = 8 * case["queries"] * case["topk"] * (2 if case["k1"] else 1)
        if kind == "exact":
            return {"bytes": 4 * d * (rows + nv) + out, "flops": 2 * nv * rows * d}
        # a query's views fall in its class's lists: those of the batch's classes are read once, in the store's type,
        # and once more as FP32 for the candidates that are rescored
        share = min(1.0, case["queries"] / case["classes"])
        eb = {"f32": 4, "bf16": 2, "fp8": 1}[case["storage"]]
        cand = min(rows * share, case["queries"] * case["rescore"] * case["views"])
        pairs = nv * case["ma"] * rows / case["codewords"]
        sif = 8 * case["queries"] * case["k1"] ** 2
        return {"bytes": 4 * d * (nv + case["codewords"]) + rows * share * d * eb + 4 * d * cand + out + sif,
                "flops": 2 * d * (nv * case["codewords"] + pairs)}
    if kind == "rerank":
        n = case["queries"] * case["k1"] ** 2
        return {"bytes": 8 * (case["queries"] * (case["cand"] + case["topk"]) + n), "flops": 2 * n}
    if kind == "aca":
        rows = 2 * case["queries"] * case["k1"] * case["k2"]
        n = rows * 2 * case["k1"] * case["k2"]
        return {"bytes": 8 * (case["queries"] * (2 * case["cand"] + case["topk"]) + rows + n), "flops": 2 * n}
    if kind in ("forward", "backward", "step"):
        nq, nr, np_ = _query_rows(case), case["shapes"] * case["views"], case["shapes"]
        di, do, eb = case["din"], case["dout"], 2 if case["dtype"] == "bf16" else 4
        project = 2 * (nq + nr) * di * do
        inputs = eb * ((nq + nr) * di + di * do)
        fwd = {"bytes": inputs + 4 * case["queries"] * np_ + 2 * nq * np_, "flops": project + 2 * nq * nr * do}
        bwd = {"bytes": inputs + 4 * ((nq + nr) * di + di * do) + 4 * case["queries"] * np_ + 2 * nq * np_,
               "flops": 3 * project + 4 * nq * np_ * do}
        if kind == "step":
            return {k: fwd[k] + bwd[k] for k in fwd}
        return fwd if kind == "forward" else bwd
    if kind == "kmeans":
        n, d, k = case["rows"], case["dim"], case["codewords"]
        return {"bytes": 4 * d * (n * case["iters"] + k), "flops": case["iters"] * (2 * n * k * d + 2 * n * d)}
    views = case["meshes"] * case["n_az"] * case["n_el"]
    tris = 2 * case["n_lon"] * (case["n_lat"] - 1)
    return {"bytes": 4 * views * case["side"] ** 2 + 24 * case["meshes"] * tris, "flops": 60 * views * tris}


# ---------------------------------------------------------------- 64 bits
def _codes64(x, cb, ma):
    """The ma nearest codewords of every row: the few nearest by FP32 scores, decided by 64-bit distances."""
    few = min(cb.shape[0], ma + 3)
    half = 0.5 * (cb * cb).sum(1)
    cb64 = cb.double()
    out = torch.empty((x.shape[0], ma), dtype=torch.int64, device="cuda")
    step = max(1, (1 << 26) // (few * x.shape[1]))
    for s in range(0, x.shape[0], step):
        c = x[s:s + step]
        near = (c @ cb.T - half).topk(few, dim=1).indices.sort(1).values
        dist = ((c.double()[:, None] - cb64[near]) ** 2).sum(2)
        out[s:s + step] = near.gather(1, dist.sort(dim=1, stable=True).indices[:, :ma])
    return out


def _exact_query(case, seed):
    """Scores of the best shapes by Eq. 4 (Eq. 3 when kind is exact): FP32 scores choose, 64 bits decide."""
    nv, rows, d = _query_rows(case), case["shapes"] * case["views"], case["dim"]
    keep = min(case["shapes"], case["topk"] + 32)
    if 2 * nv * rows * d / 5e13 + 2 * nv * keep * case["views"] * d / 8e11 + 5e-10 * rows * d > 17:
        return None  # too long in 64 bits
    db, q, offs, cb = _query_inputs(case, seed)
    n, v, b = case["shapes"], case["views"], case["queries"]
    vq = torch.from_numpy(np.repeat(np.arange(b), np.diff(offs))).cuda()
    count = torch.from_numpy(np.diff(offs)).cuda().double()
    fif = case["kind"] == "query"
    if fif:
        qc, dc = _codes64(q, cb, case["ma"]), _codes64(db, cb, 1)[:, 0]

    def reached(qcode, dcode):
        hit = qcode[:, :1] == dcode
        for a in range(1, qcode.shape[1]):
            hit |= qcode[:, a:a + 1] == dcode
        return hit

    score = torch.empty((b, n), device="cuda")
    step = max(1, (1 << 29) // (q.shape[0] * v))
    for s in range(0, n, step):
        at = slice(s * v, min(n, s + step) * v)
        sim = q @ db[at].T
        if fif:
            sim.mul_(reached(qc, dc[at]))
        best = sim.view(q.shape[0], -1, v).amax(2)
        score[:, s:s + step] = torch.zeros((b, best.shape[1]), device="cuda").index_add_(0, vq, best)
    score /= count[:, None]
    near = score.topk(keep, dim=1).indices
    out = torch.empty((b, keep), dtype=torch.float64, device="cuda")
    inner = torch.arange(v, device="cuda")
    for i in range(b):
        at = (near[i][:, None] * v + inner).reshape(-1)
        view = slice(int(offs[i]), int(offs[i + 1]))
        sim = _unit(q[view].double()) @ _unit(db[at].double()).T
        if fif:
            sim.mul_(reached(qc[view], dc[at]))
        out[i] = sim.view(sim.shape[0], keep, v).amax(2).mean(0)
    scores = out.sort(1, descending=True).values[:, :case["topk"]]
    if case["topk"] > keep:
        scores = torch.nn.functional.pad(scores, (0, case["topk"] - keep), value=-math.inf)
    if not case["k1"]:
        return {"ids": None, "scores": scores}
    # the re-rank of a query's own ranked list has no value of its own: near ties move shapes in that list
    return {"ids": None, "scores": scores, "rerank_ids": None, "rerank_scores": None}


def _best(sprime, tie, k):
    """The k largest S' of a row by (S', S, lower id)."""
    order = torch.argsort(tie, descending=True, stable=True)
    order = order[torch.argsort(sprime[order], descending=True, stable=True)]
    return sprime[order[:k]]


def _exact_rerank(case, seed):
    n, k1 = case["shapes"], case["k1"]
    ids, sc = _neighbours(n, case["classes"], k1, _gen(seed, 6))
    cid, csc = _neighbours(n, case["classes"], case["cand"], _gen(seed, 7), False, case["queries"])
    ids, sc, cid, csc = ids.long(), sc.double(), cid.long(), csc.double()
    norm = sc.sum(1)
    out = torch.empty((case["queries"], min(case["topk"], n)), dtype=torch.float64, device="cuda")
    for b in range(case["queries"]):
        fq = torch.zeros(n, dtype=torch.float64, device="cuda")
        fq[cid[b, :k1]] = csc[b, :k1]
        num = torch.minimum(fq[ids], sc).sum(1)
        tie = torch.full((n,), -math.inf, dtype=torch.float64, device="cuda")
        tie[cid[b]] = csc[b]
        out[b] = _best(num / (fq.sum() + norm - num), tie, case["topk"])
    return {"ids": None, "scores": out}


def _exact_aca(case, seed):
    n, k1, k2 = case["shapes"], case["k1"], case["k2"]
    nbr, cand = [], []
    for m in range(2):
        i, s = _neighbours(n, case["classes"], k1, _gen(seed, 10 * m + 1))
        nbr.append((i.long(), s.double()))
        i, s = _neighbours(n, case["classes"], case["cand"], _gen(seed, 10 * m + 2), False, case["queries"])
        cand.append((i.long(), s.double()))

    def fused(first):
        """Eq. 11 then Eq. 9: rows of activations, from each row's first k2 neighbours under both measures."""
        f = 0
        for m in range(2):
            src = first[1 - m]
            a = torch.zeros((src.shape[0], n), dtype=torch.float64, device="cuda")
            a.scatter_add_(1, nbr[m][0][src].reshape(src.shape[0], -1), nbr[m][1][src].reshape(src.shape[0], -1) / k2)
            f = f + 0.5 * a.sqrt_()
        return f.square_()

    fp = fused([nbr[m][0][:, :k2] for m in range(2)])
    fq = fused([cand[m][0][:, :k2] for m in range(2)])
    norm = fp.sum(1)
    out = torch.empty((case["queries"], min(case["topk"], n)), dtype=torch.float64, device="cuda")
    for b in range(case["queries"]):
        cols = fq[b].nonzero()[:, 0]  # a column that is zero in the query adds nothing to the minima
        num = torch.minimum(fp[:, cols], fq[b, cols]).sum(1)
        tie = torch.full((n,), -math.inf, dtype=torch.float64, device="cuda")
        tie[cand[0][0][b]] = cand[0][1][b]
        out[b] = _best(num / (fq[b].sum() + norm - num), tie, case["topk"])
    return {"ids": None, "scores": out}


def _mean_by_query(x, offs):
    vq = torch.from_numpy(np.repeat(np.arange(len(offs) - 1), np.diff(offs))).cuda()
    count = torch.from_numpy(np.diff(offs)).cuda().to(x.dtype)
    return torch.zeros((len(offs) - 1, x.shape[1]), dtype=x.dtype, device="cuda").index_add_(0, vq, x) / count[:, None]


def _exact_match(case, seed):
    nq, nr, di, do = _query_rows(case), case["shapes"] * case["views"], case["din"], case["dout"]
    if (6 * (nq + nr) * di * do + 2 * nq * nr * do) / 9e11 > 17:
        return None  # too long in 64 bits
    q, offs, p, w, g = _match_inputs(case, seed)
    kind = case["kind"]
    real = torch.float64
    if kind == "backward":
        arg = _argmax(q, p, w, torch.float32)[1]
        scores = None
    else:
        best, arg = _argmax(q, p, w, real)
        scores = _mean_by_query(best, offs)
        if kind == "forward":
            return {"scores": scores, "argmax": None}
    shapes, views, _ = p.shape
    q64, w64 = q.to(real), w.to(real)
    u = q64 @ w64.T
    ul = u.norm(dim=1, keepdim=True)
    v = torch.cat([c.reshape(-1, di).to(real) @ w64.T for c in p.split(256)])
    vl = v.norm(dim=1, keepdim=True)
    u, v = u / ul, v / vl
    vq = torch.from_numpy(np.repeat(np.arange(len(offs) - 1), np.diff(offs))).cuda()
    coef = g.to(real)[vq] / torch.from_numpy(np.diff(offs)).cuda().to(real)[vq, None]
    row = arg.long() + views * torch.arange(shapes, device="cuda")
    gu = torch.zeros_like(u)
    gv = torch.zeros_like(v)
    for s in range(shapes):  # one shape at a time: its views' rows are picked and added by a one-hot product
        pick = torch.nn.functional.one_hot(row[:, s] - s * views, views).to(real) * coef[:, s:s + 1]
        at = slice(s * views, (s + 1) * views)
        gu += pick @ v[at]
        gv[at] = pick.T @ u
    du = (gu - (gu * u).sum(1, keepdim=True) * u) / ul
    dv = (gv - (gv * v).sum(1, keepdim=True) * v) / vl
    dw = du.T @ q64
    for c, x in zip(dv.split(256 * views), p.split(256)):
        dw += c.T @ x.reshape(-1, di).to(real)
    dp = torch.cat([c @ w64 for c in dv.split(1 << 16)]).view(p.shape)
    grads = {"dw": dw, "dq": du @ w64, "dp": dp}
    return grads if kind == "backward" else {"scores": scores, **grads}


def _exact_kmeans(case, seed):
    s = prepare(case, seed)
    x = s["x"].double()
    cb = s["x"][torch.from_numpy(s["init"]).cuda()].clone()
    for _ in range(case["iters"]):
        c64 = cb.double()  # every step starts from float32 centres
        near = torch.cat([(a @ c64.T - 0.5 * (c64 * c64).sum(1)).argmax(1) for a in x.split(8192)])
        pick = torch.nn.functional.one_hot(near, case["codewords"]).double().T
        size = pick.sum(1, keepdim=True)
        mean = (pick @ x) / size.clamp_min(1.0)
        empty = (size[:, 0] == 0).nonzero()[:, 0]
        if len(empty):
            far = ((x - c64[near]) ** 2).sum(1).sort(descending=True, stable=True).indices
            mean[empty] = x[far[:len(empty)]]
        cb = mean.float()
    return cb.double()


def _exact_render(case, seed):
    verts, tris, vo, to = _mesh_inputs(case, seed)
    m, h, nv, d64 = case["meshes"], case["side"], case["n_az"] * case["n_el"], torch.float64
    x = verts.to(d64).view(m, -1, 3)
    t = tris.long().view(m, -1, 3)
    corner = x[torch.arange(m, device="cuda")[:, None, None], t]
    cross = torch.linalg.cross(corner[:, :, 1] - corner[:, :, 0], corner[:, :, 2] - corner[:, :, 0])
    area = 0.5 * cross.norm(dim=2, keepdim=True)
    x = x - ((area * corner.mean(2)).sum(1) / area.sum(1))[:, None]
    x = x / x.norm(dim=2).amax(1)[:, None, None]
    el = math.pi * ((torch.arange(case["n_el"], dtype=d64) + 0.5) / case["n_el"] - 0.5)
    az = 2 * math.pi * torch.arange(case["n_az"], dtype=d64) / case["n_az"]
    el, az = (a.reshape(-1).cuda() for a in torch.meshgrid(el, az, indexing="ij"))
    f = torch.stack([-el.cos() * az.cos(), -el.cos() * az.sin(), -el.sin()], 1)
    r = torch.stack([f[:, 1], -f[:, 0], 0 * az], 1)
    r = r / r.norm(dim=1, keepdim=True)
    frame = torch.stack([r, torch.linalg.cross(r, f), f], 1)  # [view, axis, 3]
    out = torch.full((m, nv, h * h), 2.0, dtype=d64, device="cuda")
    for k in range(m):
        # a mesh's triangles in every view, then one row per pixel of each one's box
        p = torch.einsum("vac,nc->vna", frame, x[k])[:, t[k]].reshape(-1, 3, 3)  # [view * tri, corner, axis]
        twice = (p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1]) - (p[:, 1, 1] - p[:, 0, 1]) * (p[:, 2, 0] - p[:, 0, 0])
        p = torch.where((twice < 0)[:, None, None], p[:, [0, 2, 1]], p)
        twice = twice.abs()
        col = (p[:, :, 0] + 1) * 0.5 * h - 0.5
        line = (1 - p[:, :, 1]) * 0.5 * h - 0.5
        j0, i0 = (a.amin(1).ceil().long().clamp(0, h) for a in (col, line))
        wide, high = (a.amax(1).floor().long().clamp(-1, h - 1) - b + 1 for a, b in ((col, j0), (line, i0)))
        box = wide.clamp_min(0) * high.clamp_min(0) * (twice > 0)
        which = torch.repeat_interleave(torch.arange(box.numel(), device="cuda"), box)
        at = torch.arange(which.numel(), device="cuda") - (box.cumsum(0) - box)[which]
        i, j = i0[which] + at // wide[which], j0[which] + at % wide[which]
        px, py = -1 + (2 * j + 1).to(d64) / h, 1 - (2 * i + 1).to(d64) / h
        c = p[which]
        edge = [(c[:, b, 0] - c[:, a, 0]) * (py - c[:, a, 1]) - (c[:, b, 1] - c[:, a, 1]) * (px - c[:, a, 0])
                for a, b in ((1, 2), (2, 0), (0, 1))]
        z = sum(e * c[:, n, 2] for n, e in enumerate(edge)) / twice[which] + 1
        inside = (edge[0] >= 0) & (edge[1] >= 0) & (edge[2] >= 0)
        view = which // t.shape[1]
        out[k].view(-1).scatter_reduce_(0, (view * h * h + i * h + j)[inside], z[inside].clamp(0, 2), "amin")
    return out.view(m, nv, h, h)


def exact(case, seed):
    kind = case["kind"]
    if kind in ("query", "exact"):
        return _exact_query(case, seed)
    if kind == "rerank":
        return _exact_rerank(case, seed)
    if kind == "aca":
        return _exact_aca(case, seed)
    if kind in ("forward", "backward", "step"):
        return _exact_match(case, seed)
    return _exact_kmeans(case, seed) if kind == "kmeans" else _exact_render(case, seed)
