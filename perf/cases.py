"""The work a user has this framework do, as cases that can be timed and compared.

A case is a dict of plain values.  Its "kind" names the entry point:

  prune    ccpm.prune: one template over a resident graph, end to end (LCC to
           its fixpoint, the non-local constraints, the final exact search),
           or with "lcc_only" the first LCC fixpoint alone
  batch    ccpm.prune_batch: many edit variants of one template
  explore  ccpm.explore: an over-constrained template relaxed edge by edge
  matches  Result.matches: participation counts of every vertex and entry
  noalloc  ccpm.lcc_fixpoint_noalloc: LCC without device allocations
  wide     ccpm.lcc_wide: LCC for up to 64 template vertices, edge labels
  order    ordering.train and Mlp.forward: the network that orders constraints

Graphs are R-MAT graphs (skew .57/.19/.19/.05) of n vertices and m CSR entries
(two per edge); neither need be round.  Labels follow the degree (its bit
length) or Zipf's law (exponent 1.2, 64 labels).  Zipf templates carry labels
of the law's tail (ranks 16 to 63), as full prunes over the frequent ones match
more than 10^12 times; the LCC phase alone also runs on frequent ones.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1912_08453_gb300 import ccpm, ordering
from paper_1912_08453_gb300 import workloads as wl

DEVICE = "cuda:0"
COUNT_CAP = 1 << 16          # matches counted before a prune reports the count as capped

# the templates of this repository's own workloads and tests
TEMPLATES = {
    "treetri6": ([5, 4, 8, 7, 4, 5], [(0, 1), (1, 2), (1, 3), (3, 4), (3, 5), (2, 3)]),
    "tree6": ([11, 3, 6, 8, 7, 9], [(0, 1), (1, 2), (1, 3), (3, 4), (4, 5)]),
    "c4tri6": ([5, 12, 11, 11, 5, 7], [(0, 1), (1, 2), (2, 3), (3, 0), (2, 4), (3, 4), (4, 5)]),
    "tree5": ([5, 4, 6, 3, 2], [(0, 1), (1, 2), (1, 3), (3, 4)]),
    "cycle5x8": ([20, 30, 40, 20, 30, 50, 60, 40],
                 [(0, 1), (1, 2), (2, 3), (3, 4), (4, 0), (4, 5), (5, 6), (6, 7), (2, 7)]),
    "cycle5x8_frequent": ([0, 1, 2, 0, 1, 3, 4, 2],
                          [(0, 1), (1, 2), (2, 3), (3, 4), (4, 0), (4, 5), (5, 6), (6, 7), (2, 7)]),
    "c4tri7": ([20, 30, 40, 20, 50, 60, 30], [(0, 1), (1, 2), (2, 3), (3, 0), (2, 4), (3, 4), (4, 5), (5, 6)]),
    "clique5": ([6, 7, 6, 7, 8],
                [(0, 1), (0, 2), (0, 3), (0, 4), (1, 2), (1, 3), (1, 4), (2, 3), (2, 4), (3, 4)]),
    "c4chord5": ([5, 6, 5, 6, 7], [(0, 1), (1, 2), (2, 3), (3, 0), (0, 2), (3, 4)]),
}


def listed():
    return [
        # the smallest call: an interactive query on a graph of a few thousand vertices
        {"name": "prune_4k", "kind": "prune", "n": 4096, "m": 90000, "labels": "degree", "template": "treetri6"},
        # an ordinary small graph: a tree with a triangle, cycle constraint and final count
        {"name": "prune_64k", "kind": "prune", "n": 65536, "m": 1700002, "labels": "degree", "template": "treetri6"},
        # an acyclic template on a large graph: LCC does nearly everything
        {"name": "prune_tree_4m", "kind": "prune", "n": 1 << 22, "m": 128000000, "labels": "degree", "template": "tree6"},
        # a 4-cycle and a triangle on a large graph of ragged size: LCC, then non-local walks
        {"name": "prune_cycles_3m", "kind": "prune", "n": 3000001, "m": 89999998, "labels": "degree", "template": "c4tri6"},
        # repeated labels and a 5-cycle (template-driven search constraints), capped count
        {"name": "prune_tds_16m", "kind": "prune", "n": 1 << 24, "m": 500000000, "labels": "zipf", "template": "cycle5x8"},
        # the LCC phase where half of the vertices start active, on the largest graph
        {"name": "lcc_frequent_32m", "kind": "prune", "n": 1 << 25, "m": 1000000000, "labels": "zipf",
         "template": "cycle5x8_frequent", "lcc_only": True},
        # exploratory search over one resident graph: edit variants of one query, pruned side by side
        {"name": "batch_4m", "kind": "batch", "n": 1 << 22, "m": 124000000, "labels": "zipf", "template": "c4tri7",
         "count": 24, "variants": 5, "workers": 8},
        # an over-constrained clique relaxed until some variant matches
        {"name": "explore_8k", "kind": "explore", "n": 8192, "m": 190002, "labels": "degree", "template": "clique5",
         "max_removed": 3},
        # which vertices and edges take part in how many matches, after a prune
        {"name": "matches_1m", "kind": "matches", "n": 1 << 20, "m": 30000000, "labels": "degree", "template": "c4tri6"},
        # LCC inside a caller that may not allocate, near the largest graph it takes
        {"name": "noalloc_250k", "kind": "noalloc", "n": 249999, "m": 6900002, "labels": "degree", "template": "tree5"},
        # a 48-vertex template with edge labels
        {"name": "wide_4m", "kind": "wide", "n": 1 << 22, "m": 124000000, "labels": "degree", "n0": 48, "extra": 6,
         "edge_labels": 3},
        # training of the ordering network on logged constraints, then the scores of new ones
        {"name": "order_train", "kind": "order", "records": 11452, "steps": 100, "batch": 256, "score": 64},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["prune", "prune", "prune", "lcc", "lcc", "batch", "explore", "matches", "noalloc", "wide",
                       "order"])

    def sized(kind, lo, hi, **more):
        n = size(lo, hi)
        return {"kind": kind, "n": n, "m": 2 * int(n * rng.uniform(7.0, 15.0)), **more}

    if kind == "prune":
        if rng.random() < 0.5:
            return sized("prune", 3000, 1 << 22, labels="degree",
                         template=rng.choice(["treetri6", "tree6", "c4tri6", "tree5"]))
        return sized("prune", 30000, 1 << 23, labels="zipf", template=rng.choice(["cycle5x8", "c4tri7"]),
                     shift=rng.randint(-4, 3))
    if kind == "lcc":
        return sized("prune", 30000, 1 << 24, labels="zipf", lcc_only=True, random_template=rng.randint(1, 10**6),
                     n0=rng.randint(3, 12), extra=rng.randint(0, 4), used=rng.randint(4, 12))
    if kind == "batch":
        return sized("batch", 30000, 1 << 21, labels="zipf", template="c4tri7", count=rng.randint(4, 24),
                     variants=rng.randint(1, 10**6), workers=rng.choice([2, 4, 8]))
    if kind == "explore":
        return sized("explore", 3000, 40000, labels="degree", template=rng.choice(["clique5", "c4chord5"]),
                     max_removed=rng.randint(1, 3))
    if kind == "matches":
        return sized("matches", 10000, 1 << 20, labels="degree", template=rng.choice(["treetri6", "tree6", "c4tri6"]))
    if kind == "noalloc":
        return sized("noalloc", 3000, 250000, labels="degree", template=rng.choice(["tree5", "treetri6", "c4tri6"]))
    if kind == "wide":
        return sized("wide", 30000, 1 << 21, labels="degree", n0=rng.randint(20, 64), extra=rng.randint(0, 8),
                     edge_labels=rng.randint(1, 4))
    return {"kind": "order", "records": size(500, 12000), "steps": rng.randint(40, 110), "batch": size(60, 512),
            "score": rng.randint(1, 64)}


# ------------------------------------------------------------------ inputs

def _graph(case, seed):
    n, edges = case["n"], case["m"] // 2
    scale = (n - 1).bit_length()
    factor = math.ceil(1.03 * edges / (n * (n / (1 << scale))))
    while True:
        src, dst = wl.rmat_edges_philox(scale, factor, seed=seed, device=DEVICE)
        low, high = torch.minimum(src, dst), torch.maximum(src, dst)
        del src, dst
        key = torch.unique((low * n + high)[(low < high) & (high < n)])
        del low, high
        if key.numel() >= edges:
            break
        factor += max(1, factor // 4)
    # as many edges as asked for, spread evenly over those drawn
    key = key[torch.arange(edges, device=DEVICE) * key.numel() // edges]
    low = torch.div(key, n, rounding_mode="floor")
    row_ptr, col = wl.csr_from_edges_torch(n, low, key - low * n)
    del key, low
    if case["labels"] == "degree":
        labels = wl.degree_labels_torch(row_ptr)
    else:
        labels = wl.zipf_labels_philox(n, seed=seed + 7, device=DEVICE)
    return row_ptr, col, labels


def _template(case):
    if "random_template" in case:
        t = wl.random_template(case["random_template"], case["n0"], case["extra"], range(case["used"]))
        return t.labels, t.edges
    labels, edges = TEMPLATES[case["template"]]
    return [x + case.get("shift", 0) for x in labels], edges


def _sampled_template(case, seed, row_ptr, col, labels, edge_labels):
    """A breadth-first sample of the graph (so that it matches): its vertices'
    labels, the walk's tree edges and a few more edges among them, with their
    edge labels."""
    rng = np.random.default_rng(seed)
    while True:
        order, tree = [int(rng.integers(case["n"]))], []
        rows = {}
        for v in order:
            b, e = int(row_ptr[v]), int(row_ptr[v + 1])
            rows[v] = (col[b:e].cpu().numpy(), edge_labels[b:e].cpu().numpy())
            if len(order) < case["n0"]:
                new = np.setdiff1d(rows[v][0], order)[: case["n0"] - len(order)]
                tree += [(v, int(u)) for u in new]
                order += [int(u) for u in new]
        if len(order) == case["n0"]:
            break
    at = {v: i for i, v in enumerate(order)}
    known = {(v, int(u)): int(x) for v in order for u, x in zip(*rows[v]) if int(u) in at}
    tree_set = {frozenset(e) for e in tree}
    chords = [e for e in sorted(known) if e[0] < e[1] and frozenset(e) not in tree_set]
    rng.shuffle(chords)
    edges = tree + [tuple(int(x) for x in e) for e in chords[: case["extra"]]]
    return ([int(labels[v]) for v in order], [tuple(sorted((at[a], at[b]))) for a, b in edges],
            [known[e] for e in edges])


def _order_data(case, seed):
    """Logged constraints as the pipeline leaves them (kind, sizes, candidate
    counts on a log scale) and their targets, minus the log2 of a cost."""
    rng = np.random.default_rng(seed)

    def features(rows):
        x = np.zeros((rows, ccpm.MLP_IN), dtype=np.float32)
        x[np.arange(rows), rng.integers(0, 5, rows)] = 1.0
        x[:, 5:8] = rng.integers(3, 10, (rows, 3)) / 8.0
        x[:, 8:12] = np.sort(rng.uniform(0.1, 0.8, (rows, 4)), axis=1)
        x[:, 12] = rng.uniform(0.3, 1.0, rows)
        x[:, 13] = rng.integers(0, 4, rows) / 4.0
        x[:, 14] = rng.uniform(0.0, 1.0, rows)
        x[:, 15] = rng.uniform(0.2, 0.8, rows)
        return x

    x, new = features(case["records"]), features(case["score"])
    cost = 6.0 + 6.0 * x[:, 11] + x[:, 6] + 0.3 * rng.standard_normal(case["records"])
    return x, (-cost).astype(np.float32), new


def prepare(case, seed):
    stream = torch.cuda.Stream()
    ctx = ccpm.Context(0, stream=stream.cuda_stream)
    s = {"case": case, "stream": stream, "ctx": ctx}
    if case["kind"] == "order":
        s["x"], s["y"], s["new"] = _order_data(case, seed)
        s["seed"] = seed
        return s
    row_ptr, col, labels = _graph(case, seed)
    n, words = case["n"], (case["m"] + 31) // 32
    if case["kind"] == "wide":
        el = wl.edge_labels(row_ptr, col, case["edge_labels"], seed=seed, weights=[8, 1, 1, 1][: case["edge_labels"]])
        s["template"] = _sampled_template(case, seed, row_ptr, col, labels, el)
    torch.cuda.synchronize()
    if case["kind"] == "noalloc":
        s["csr"], s["template"] = (row_ptr, col, labels), _template(case)
    else:
        s["graph"] = ccpm.Graph(ctx, row_ptr, col, labels)
    if case["kind"] == "wide":
        s["graph"].set_edge_labels(el)
        return s
    if case["kind"] == "batch":
        base = wl.Template(*_template(case), name="base")
        pool = sorted(set(base.labels))
        every = [base] + wl.edit_variants(base, case["count"] - 1, seed=case["variants"], label_pool=pool)
        s["templates"] = [ccpm.Template(ctx, t.labels, t.edges) for t in every]
        s["results"] = None
        s["options"] = ccpm.options(max_embeddings=COUNT_CAP, batch_workers=case["workers"])
    elif case["kind"] != "noalloc":
        s["template"] = ccpm.Template(ctx, *_template(case))
        s["result"] = None
        s["options"] = ccpm.options(max_embeddings=COUNT_CAP, lcc_only=int(case.get("lcc_only", False)))
    if case["kind"] == "matches":
        s["result"] = ccpm.prune(ctx, s["graph"], s["template"])
        return s
    rows = case["count"] if case["kind"] == "batch" else 1
    s["omega"] = torch.empty((rows, n), dtype=torch.int32, device=DEVICE)
    s["bits"] = torch.empty((rows, words), dtype=torch.int32, device=DEVICE)
    torch.cuda.synchronize()
    return s


# -------------------------------------------------------------------- runs

def _read(s, row, r):
    """What a caller reads of a pruned template."""
    r.omega(s["omega"][row])
    r.edge_bitmap(s["bits"][row])
    c = r.counts()
    return [c["match_embeddings"], c["count_valid"], c["active_v"], c["active_e_dir"], c["edges_scanned_lcc"],
            *r.phase_rounds()]


def run(s):
    kind, ctx = s["case"]["kind"], s["ctx"]
    if kind == "order":
        c = s["case"]
        net = ordering.train(ctx, s["x"], s["y"], steps=c["steps"], batch=c["batch"], seed=s["seed"])
        out = {"params": net.params(), "scores": net.forward(s["new"])}
        net.close()
        return out
    with torch.cuda.stream(s["stream"]):
        if kind == "prune":
            s["result"] = ccpm.prune(ctx, s["graph"], s["template"], s["options"], result=s["result"],
                                     allow_budget=True)
            return {"counts": _read(s, 0, s["result"]), "omega": s["omega"], "bits": s["bits"]}
        if kind == "batch":
            s["results"] = ccpm.prune_batch(ctx, s["graph"], s["templates"], s["options"], results=s["results"],
                                            allow_budget=True)
            counts = [_read(s, i, r)[:5] for i, r in enumerate(s["results"])]
            return {"counts": np.asarray(counts, dtype=np.int64), "omega": s["omega"], "bits": s["bits"]}
        if kind == "explore":
            level, union, variants, _ = ccpm.explore(ctx, s["graph"], s["template"], s["case"]["max_removed"],
                                                     s["options"], allow_budget=True)
            union.omega(s["omega"][0])
            union.edge_bitmap(s["bits"][0])
            union.close()
            table = np.zeros((256, 5), dtype=np.int64)        # as many as a 5-clique has, and more
            for row, v in zip(table, variants):
                row[:] = v["level"], v["removed"], v["active_v"], v["active_e_dir"], v["match_embeddings"]
            return {"level": level, "variants": table, "omega": s["omega"], "bits": s["bits"]}
        if kind == "matches":
            count, _, vertices, entries = s["result"].matches(s["template"], vertex_counts=True, entry_counts=True,
                                                              device=True)
            return {"count": count, "vertices": vertices, "entries": entries}
        if kind == "noalloc":
            rounds, scanned = ccpm.lcc_fixpoint_noalloc(0, *s["csr"], *s["template"], s["omega"][0], s["bits"][0],
                                                        stream=s["stream"].cuda_stream)
            return {"rounds": rounds, "scanned": scanned, "omega": s["omega"], "bits": s["bits"]}
        omega, bits, stats = ccpm.lcc_wide(ctx, s["graph"], *s["template"], device_out=True)
        return {"omega": omega, "bits": bits, "rounds": stats["rounds"], "scanned": stats["edges_scanned"],
                "vertices": stats["vertices_scanned"]}


# ------------------------------------------------------ what it has to move

# share of an R-MAT graph's entries that lie in the rows of one degree class
# (bit length 1 to 16 of the degree); the classes swing with the scale, these
# are means over scales 12 to 20
_DEGREE_SHARE = [0, .005, .012, .024, .046, .060, .113, .136, .131, .143, .138, .114, .03, .03, .02, .004, .001]


def work(case):
    """Bytes every pass needs: each vertex's label, the offsets and the columns
    of the rows whose vertex carries a label of the template, and the results.
    Batches and explorations read the graph once for all of their templates."""
    if case["kind"] == "order":
        per_row = 2 * (16 * 64 + 64 * 64 + 64)
        rows = case["steps"] * case["batch"]
        return {"bytes": 68.0 * rows + 4.0 * ccpm.MLP_PARAMS, "flops": 3.0 * per_row * rows}
    n, m = case["n"], case["m"]
    if case["kind"] == "wide":
        share, out = 0.9, 8.0 * n + m / 8
        per_entry = 5.0
    else:
        labels = set(_template(case)[0])
        if case["labels"] == "zipf":
            total = sum((k + 1.0) ** -1.2 for k in range(64))
            share = sum((k + 1.0) ** -1.2 for k in labels) / total
        else:
            share = sum(_DEGREE_SHARE[k] for k in labels)
        per_entry = 4.0
        out = case.get("count", 1) * (4.0 * n + m / 8)
    if case["kind"] == "matches":
        share, out = 0.0, 8.0 * (n + m) + 4.0 * n
    return {"bytes": n + share * (8.0 * n + per_entry * m) + out, "flops": 0.0}


# --------------------------------------------------------- 64-bit reference

def _splitmix(z):
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    return z ^ (z >> np.uint64(31))


def exact(case, seed):
    """The training in 64 bits (every other kind returns whole numbers)."""
    if case["kind"] != "order":
        return None
    x, y, new = (a.astype(np.float64) for a in _order_data(case, seed))
    step = np.uint64(0x9E3779B97F4A7C15)
    with np.errstate(over="ignore"):
        u = _splitmix(np.uint64(seed) + step * np.arange(1, 16 * 64 + 64 * 64 + 64 + 1, dtype=np.uint64))
        u = (u >> np.uint64(11)).astype(np.float64) / 2.0 ** 53
        sample = _splitmix(np.uint64(seed) + step * np.arange(1, case["steps"] * case["batch"] + 1, dtype=np.uint64))
    sample = (sample % np.uint64(case["records"])).astype(np.int64).reshape(case["steps"], case["batch"])
    cut = [16 * 64, 16 * 64 + 64 * 64]
    w1, w2, w3 = (((2 * v - 1) * math.sqrt(6.0 / f)).astype(np.float32).astype(np.float64)
                  for v, f in zip(np.split(u, cut), (16, 64, 64)))
    p = [w1.reshape(16, 64), np.zeros(64), w2.reshape(64, 64), np.zeros(64), w3, np.zeros(1)]
    m, v = [np.zeros_like(a) for a in p], [np.zeros_like(a) for a in p]
    lr, b1, b2 = 2e-3, 0.9, 0.999

    def forward(a):
        z1 = a @ p[0] + p[1]
        h1 = np.maximum(z1, 0)
        z2 = h1 @ p[2] + p[3]
        h2 = np.maximum(z2, 0)
        return z1, h1, z2, h2, h2 @ p[4] + p[5]

    for t in range(case["steps"]):
        a = x[sample[t]]
        z1, h1, z2, h2, out = forward(a)
        d = (out - y[sample[t]]) / case["batch"]
        d2 = d[:, None] * p[4] * (z2 > 0)
        d1 = (d2 @ p[2].T) * (z1 > 0)
        grad = [a.T @ d1, d1.sum(0), h1.T @ d2, d2.sum(0), h2.T @ d, d.sum(keepdims=True)]
        for i, g in enumerate(grad):
            m[i] = b1 * m[i] + (1 - b1) * g
            v[i] = b2 * v[i] + (1 - b2) * g * g
            p[i] = p[i] - lr * (m[i] / (1 - b1 ** (t + 1))) / (np.sqrt(v[i] / (1 - b2 ** (t + 1))) + 1e-8)
    return {"params": np.concatenate([a.reshape(-1) for a in p]), "scores": forward(new)[4]}
