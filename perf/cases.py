"""The work this engine is used for, as cases that can be timed one by one.

A case names a way of calling the engine (``kind``), a graph by its numbers and
the expressions.  Graphs are drawn on the GPU from the seed: ``er`` graphs have
uniform edges and labels (configuration 1: 1,000 vertices, 5,000 edges, 4
labels), the others are R-MAT graphs with Zipf labels (configurations 2-4).
Start vertices are drawn in proportion to their out-degree unless a case takes
consecutive ones.  One context serves all states, as in a program that loads
several graphs; its workspace and memory pool are warm after the first call.

Outputs are integers: the rows themselves where the call hands rows out (in the
caller's own buffer, whose unused end stays zero), and (count, digest sum,
digest xor) plus the work counters (product edges, product vertices) that
``result_info`` / ``result_stats`` report.
"""

from __future__ import annotations

import math

import numpy as np
import torch

from paper_2602_20748_gb300 import rpq, synth

TRIANGLE = "a;b.c*;d*"  # x -a-> y, x -b.c*-> z, y -d*-> z (configuration 3)
ALLPAIRS = "a*;(a|b)+.c;a.b*.c;(a.b)*"  # configuration 2


def listed():
    return [
        # one lookup in a small graph: the smallest call there is, all latency
        dict(name="point-er1k", kind="rows", graph="er", n=1000, edges=5000, labels=4, regex="a.b.c*", sources=1),
        # configuration 1: every pair of the small graph, fetched
        dict(name="allpairs-er1k", kind="rows", graph="er", n=1000, edges=5000, labels=4, regex="a.b.c*",
             sources=1000),
        # one lookup in a large graph (what the plain arm of configuration 4 does per query)
        dict(name="point-rmat20", kind="rows", graph="rmat", n=1 << 20, edges=1 << 24, labels=8, regex="a.b*.c",
             sources=1),
        # the entry point that allocates nothing, at its largest number of start vertices
        dict(name="static64-rmat18", kind="static", graph="rmat", n=1 << 18, edges=1 << 22, labels=8,
             regex="(a|b)+.c", sources=64),
        # a few hundred start vertices on an odd-sized graph, rows fetched
        dict(name="rows300-n65537", kind="rows", graph="rmat", n=65537, edges=1 << 20, labels=8, regex="a.(b|c)*",
             sources=300),
        # the reverse plan from a ragged number of targets, counted
        dict(name="reverse1500-rmat18", kind="count", graph="rmat", n=1 << 18, edges=1 << 22, labels=8,
             regex="a.b*.c", sources=1500, reverse=True),
        # configuration 2: one batch of 4,096 consecutive start vertices, its four expressions, rows kept on the device
        dict(name="allpairs4096-rmat20", kind="range", graph="rmat", n=1 << 20, edges=1 << 24, labels=8,
             regex=ALLPAIRS, sources=4096),
        # rows streamed into host memory while the device goes on (two batches)
        dict(name="stream8192-rmat18", kind="stream", graph="rmat", n=1 << 18, edges=1 << 22, labels=8,
             regex="b.c.d?", sources=8192),
        # a small batch of different expressions, rows fetched
        dict(name="batch48-rmat16", kind="batchrows", graph="rmat", n=1 << 16, edges=1 << 20, labels=8, sources=48),
        # configuration 4: 4,096 different expressions in one call, a summary of each
        dict(name="batch4096-rmat22", kind="batch", graph="rmat", n=1 << 22, edges=1 << 26, labels=8, sources=4096),
        # configuration 3: the triangle from 4,096 values of x, counted
        dict(name="triangle4096-rmat22", kind="crpq", graph="rmat", n=1 << 22, edges=1 << 26, labels=10, zipf=1.1,
             regex=TRIANGLE, sources=4096),
        # a triangle's tuples with a label on each variable, fetched
        dict(name="triangle-rows-er20k", kind="crpqrows", graph="er", n=20000, edges=100000, labels=4, regex=TRIANGLE,
             sources=2000, vlabels=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["rows", "rows", "static", "count", "range", "stream", "batchrows", "batch", "crpq",
                       "crpqrows"])
    rmat = kind in ("range", "crpq") or (kind != "crpqrows" and rng.random() < 0.75)
    c = dict(kind=kind, graph="rmat" if rmat else "er", labels=rng.choice([4, 6, 8, 10]))
    top = {"rows": 1 << 20, "static": 1 << 18, "count": 1 << 19, "range": 1 << 19, "stream": 1 << 18,
           "batchrows": 1 << 17, "batch": 1 << 19, "crpq": 1 << 19, "crpqrows": 20000}[kind]
    c["n"] = _log(rng, 1000 if top < (1 << 19) else 4000, top)
    c["edges"] = int(c["n"] * rng.uniform(5, 16 if rmat else 8))
    c["regex"] = rng.choice(["a.b.c*", "a.b*.c", "(a|b)+.c", "(a.b)*", "a*", "a.(b|c)*", "d.b?.c+"])
    if kind == "rows":
        c["sources"] = _log(rng, 1, max(2, min(1000, 30_000_000 // c["n"])))
    elif kind == "static":
        c["sources"] = rng.randint(1, 64)
    elif kind == "count":
        c.update(sources=_log(rng, 65, 4096), reverse=rng.random() < 0.5)
    elif kind == "range":
        c["sources"] = min(c["n"], _log(rng, 257, 4096))
    elif kind == "stream":
        c["sources"] = min(c["n"], _log(rng, 1000, 8192))
        c["regex"] = rng.choice(["b.c.d?", "c.d.e?", "b.c?"])
    elif kind == "batchrows":
        c["sources"] = _log(rng, 2, 200)
        del c["regex"]
    elif kind == "batch":
        c["sources"] = _log(rng, 16, 2000)
        del c["regex"]
    elif kind == "crpq":
        c.update(sources=_log(rng, 50, 1024), regex=TRIANGLE, zipf=1.1)
    else:
        c["sources"] = _log(rng, 50, max(100, min(2000, 10_000_000 // c["n"])))
        c.update(regex=TRIANGLE, labels=4, vlabels=rng.random() < 0.5)
    return c


_CTX = None


def _ctx():
    global _CTX
    if _CTX is None:
        _CTX = rpq.Context(device=0)
    return _CTX


def _edges(case, seed):
    """(src, dst, label) of the case's graph, int64 on the GPU, and the generator they came from."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, m, labels = case["n"], case["edges"], case["labels"]

    def rand(k):
        return torch.rand(k, generator=g, device="cuda")

    if case["graph"] == "er":
        src = torch.randint(n, (m,), generator=g, device="cuda")
        dst = torch.randint(n, (m,), generator=g, device="cuda")
        return src, dst, torch.randint(labels, (m,), generator=g, device="cuda"), g
    scale = max(1, (n - 1).bit_length())
    src = torch.zeros(m, dtype=torch.int64, device="cuda")
    dst = torch.zeros(m, dtype=torch.int64, device="cuda")
    for level in range(scale):  # quadrants (0.57, 0.19, 0.19, 0.05)
        u = rand(m)
        src |= (u >= 0.76).long() << level
        dst |= (((u >= 0.57) & (u < 0.76)) | (u >= 0.95)).long() << level
    perm = torch.randperm(1 << scale, generator=g, device="cuda")
    src, dst = perm[src] % n, perm[dst] % n
    cdf = torch.from_numpy(np.cumsum(synth.zipf_probs(labels, case.get("zipf", 1.2)))).float().cuda()
    lab = torch.searchsorted(cdf, rand(m), right=True).clamp_(max=labels - 1)
    return src, dst, lab, g


def _inputs(case, seed):
    """Host arrays of the graph, the start vertices (ascending, distinct where the call takes a set) and vertex labels."""
    src, dst, lab, g = _edges(case, seed)
    k, n = case["sources"], case["n"]
    if case["kind"] in ("range", "stream"):
        first = int(torch.randint(n - k + 1, (1,), generator=g, device="cuda"))
        starts = np.arange(first, first + k, dtype=np.uint32)
    elif k >= n:
        starts = np.arange(n, dtype=np.uint32)
    elif case["kind"] in ("crpq", "crpqrows"):  # values of variable 0: any vertices
        starts = torch.randperm(n, generator=g, device="cuda")[:k].cpu().numpy().astype(np.uint32)
    else:
        ends = dst if case.get("reverse") else src
        some = ends[torch.randint(len(ends), (64 * k,), generator=g, device="cuda")].cpu().numpy()
        _, at = np.unique(some, return_index=True)
        starts = np.sort(some[np.sort(at)[:k]]).astype(np.uint32)
    vl = torch.randint(5, (n,), generator=g, device="cuda").to(torch.uint8).cpu().numpy() if case.get("vlabels") else None
    host = [x.to(t).cpu().numpy() for x, t in ((src, torch.int32), (dst, torch.int32), (lab, torch.int16))]
    return host[0].view(np.uint32), host[1].view(np.uint32), host[2].view(np.uint16), starts, vl


def prepare(case, seed):
    ctx = _ctx()
    src, dst, lab, starts, vl = _inputs(case, seed)
    s = dict(case, ctx=ctx, starts=starts)
    s["g"] = rpq.load_graph(ctx, case["n"], case["labels"], src, dst, lab, vl)
    if case["kind"] in ("batch", "batchrows"):
        regexes, sources = synth.batch_queries(case["sources"], case["labels"], 1.2, src[:1 << 20], case["n"], seed)
        s.update(queries=[rpq.compile_rpq(ctx, r) for r in regexes], starts=sources)
        rpq.rpq_set_option(ctx, "batch_evict", 1024)  # what rpq_autotune_batch keeps for configuration 4
    else:
        s["queries"] = [rpq.compile_rpq(ctx, r) for r in case["regex"].split(";")]
    if case["kind"] in ("crpq", "crpqrows"):
        a, bc, d = s["queries"]
        s.update(atoms=[(0, a, 1), (0, bc, 2), (1, d, 2)], vl=[0, 1, 2] if vl is not None else None)
    # the caller's buffers: device memory for the call that writes there, pinned or plain host memory for the others
    k, n = len(s["starts"]), case["n"]
    if case["kind"] == "static":
        s["out"] = torch.zeros(2 * k * n, dtype=torch.int32, device="cuda")
    elif case["kind"] == "stream":
        s["out"] = np.zeros(k * min(n, 1 << 14), dtype=np.uint32)
        s["per_source"] = np.zeros(case["sources"], dtype=np.int64)
    elif case["kind"] in ("rows", "batchrows", "crpqrows"):
        values = 3 << 24 if case["kind"] == "crpqrows" else 2 * case["sources"] * n
        s["out"] = torch.zeros(values, dtype=torch.int32).pin_memory().numpy().view(np.uint32)
    return s


def _u64(*values):
    return np.array(values, dtype=np.uint64).view(np.int64)


def _info(r):
    count, _, hs, hx = rpq.result_info(r)
    st = rpq.result_stats(r)
    return _u64(count, hs, hx), _u64(st["product_edges"], st["product_vertices"])


def run(s):
    ctx, g, kind = s["ctx"], s["g"], s["kind"]
    if kind == "static":
        rows = rpq.run_rpq_static(ctx, g, s["queries"][0], s["starts"], s["out"].data_ptr(), s["out"].numel() // 2)
        return [s["out"], rows]
    if kind == "range":
        out = []
        for q in s["queries"]:
            r = rpq.run_rpq_range(ctx, g, q, int(s["starts"][0]), int(s["starts"][-1]) + 1, rpq.RPQ_MATERIALIZE)
            out += _info(r)
            r.free()
        return out
    if kind == "stream":
        st = rpq.Stream(ctx, g, s["queries"][0], int(s["starts"][0]), int(s["starts"][-1]) + 1)
        s["per_source"][:] = 0
        at = 0
        while (blk := st.next_block()) is not None:
            src, off, dst = blk
            s["out"][at:at + len(dst)] = dst
            s["per_source"][src - s["starts"][0]] += np.diff(off).astype(np.int64)
            at += len(dst)
        count, hs, hx, stats = st.info()
        st.close()
        return [s["out"].view(np.int32), s["per_source"], _u64(count, hs, hx),
                _u64(stats["product_edges"], stats["product_vertices"])]
    if kind == "rows":
        r = rpq.run_rpq(ctx, g, s["queries"][0], s["starts"], rpq.RPQ_MATERIALIZE)
    elif kind == "count":
        r = rpq.run_rpq(ctx, g, s["queries"][0], s["starts"],
                        rpq.RPQ_COUNT_ONLY | (rpq.RPQ_REVERSE if s["reverse"] else 0))
    elif kind == "batchrows":
        r = rpq.run_rpq_batch(ctx, g, s["queries"], s["starts"], rpq.RPQ_MATERIALIZE)
    elif kind == "batch":
        r = rpq.run_rpq_batch(ctx, g, s["queries"], s["starts"], rpq.RPQ_PER_QUERY)
    else:
        r = rpq.run_crpq(ctx, g, 3, s["atoms"], var_label=s["vl"], restrict0=s["starts"],
                         flags=rpq.RPQ_COUNT_ONLY if kind == "crpq" else rpq.RPQ_MATERIALIZE)
    if kind in ("rows", "batchrows", "crpqrows"):
        rows = rpq.fetch_pairs(r, max_rows=len(s["out"]) // (3 if kind == "crpqrows" else 2), out=s["out"])
        out = [s["out"].view(np.int32), len(rows)]
    elif kind == "batch":
        out = [np.array([rpq.result_query_stats(r, i) for i in range(len(s["queries"]))], np.uint64).view(np.int64)]
    else:
        out = []
    info, counters = _info(r)
    r.free()
    # the work counters of a CRPQ depend on the order its atoms are joined in
    return out + [info] if kind in ("crpq", "crpqrows") else out + [info, counters]


def work(case):
    """Bytes of one pass: per start vertex and expression, the start vertices' share of the adjacency read once (column
    ids of every edge on the expression's labels, once per 4,096 start vertices), a visited bit per (start vertex,
    state, vertex) written and read, and the rows or their bits."""
    n, m, k, kind = case["n"], case["edges"], case["sources"], case["kind"]
    if kind in ("batch", "batchrows"):
        exprs, states = 1, 5
    else:
        exprs, states = len(case["regex"].split(";")), 3
    # a single start vertex need not touch every edge: the closure of a few sources reaches a part of the graph
    share = min(1.0, 0.1 + k / 64)
    adjacency = exprs * 4.0 * m * 0.6 * share * max(1, k // 4096)
    visited = exprs * states * float(k) * n / 8 * 2 * share
    density = 0.1  # rows per (start vertex, vertex)
    rows = 4.0 * k * n * density * exprs if kind in ("range",) else 8.0 * k * n * 0.02 * share
    if kind in ("count", "batch", "crpq"):
        rows = 24.0 * k
    return {"bytes": adjacency + visited + rows, "flops": 0.0}


# ---- the rows by plain set algebra ------------------------------------------------------------------------------

def _parse(text):
    """Regex over one-letter labels -> nested tuples: ("l", id), ("cat" | "or", x, y), ("*" | "+" | "?", x)."""
    toks = [c for c in text if c not in " ."]
    pos = 0

    def alt():
        nonlocal pos
        x = cat()
        while pos < len(toks) and toks[pos] == "|":
            pos += 1
            x = ("or", x, cat())
        return x

    def cat():
        x = post()
        while pos < len(toks) and toks[pos] not in "|)":
            x = ("cat", x, post())
        return x

    def post():
        nonlocal pos
        if toks[pos] == "(":
            pos += 1
            x = alt()
        else:
            x = ("l", ord(toks[pos]) - ord("a"))
        pos += 1
        while pos < len(toks) and toks[pos] in "*+?":
            x = (toks[pos], x)
            pos += 1
        return x

    return alt()


def _image(tree, x, edges):
    """The vertices (per column of the boolean [n, k] matrix x) that a path of the expression reaches."""
    op = tree[0]
    if op == "l":
        src, dst = edges.get(tree[1], (None, None))
        y = torch.zeros(x.shape, dtype=torch.float32, device=x.device)
        if src is not None:
            for a in range(0, len(src), 1 << 20):
                y.index_add_(0, dst[a:a + (1 << 20)], x[src[a:a + (1 << 20)]].float())
        return y > 0
    if op == "cat":
        return _image(tree[2], _image(tree[1], x, edges), edges)
    if op == "or":
        return _image(tree[1], x, edges) | _image(tree[2], x, edges)
    if op == "?":
        return x | _image(tree[1], x, edges)
    seen = _image(tree[1], x, edges) if op == "+" else x
    while True:
        more = seen | _image(tree[1], seen, edges)
        if torch.equal(more, seen):
            return seen
        seen = more


def _splitmix(x):
    def shift(z, k):
        return (z >> k) & ((1 << (64 - k)) - 1)

    z = x + (0x9E3779B97F4A7C15 - (1 << 64))
    z = (z ^ shift(z, 30)) * (0xBF58476D1CE4E5B9 - (1 << 64))
    z = (z ^ shift(z, 27)) * (0x94D049BB133111EB - (1 << 64))
    return z ^ shift(z, 31)


def _xor(x):
    while len(x) > 1:
        if len(x) % 2:
            x = torch.cat([x, x.new_zeros(1)])
        x = x[0::2] ^ x[1::2]
    return x if len(x) else x.new_zeros(1)


def exact(case, seed):
    kind = case["kind"]
    if kind not in ("rows", "static", "count") or case["sources"] * case["edges"] > 1 << 33:
        return None
    src, dst, lab, starts, _ = _inputs(case, seed)
    src, dst, lab = (torch.from_numpy(x.astype(np.int64)).cuda() for x in (src, dst, lab))
    if case.get("reverse"):
        src, dst = dst, src
    edges = {i: (src[lab == i], dst[lab == i]) for i in range(case["labels"])}
    tree = _parse(case["regex"])
    if case.get("reverse"):
        def flip(t):
            return t if t[0] == "l" else ("cat", flip(t[2]), flip(t[1])) if t[0] == "cat" else (
                t[0], *(flip(x) for x in t[1:]))
        tree = flip(tree)
    ids = torch.from_numpy(starts.astype(np.int64)).cuda()
    rows = []
    for a in range(0, len(ids), 64):
        part = ids[a:a + 64]
        x = torch.zeros(case["n"], len(part), dtype=torch.bool, device="cuda")
        x[part, torch.arange(len(part), device="cuda")] = True
        at = _image(tree, x, edges).t().nonzero()
        rows.append(torch.stack([part[at[:, 0]], at[:, 1]], 1))
    rows = torch.cat(rows)
    h = _splitmix((rows[:, 0] << 32) | rows[:, 1])
    info = np.array([len(rows), int(h.sum()), int(_xor(h)[0])], dtype=np.int64)
    if kind == "count":
        return [info, None]
    out = torch.zeros(2 * case["sources"] * case["n"], dtype=torch.int32, device="cuda")
    out[: 2 * len(rows)] = rows.to(torch.int32).reshape(-1)
    return [out, len(rows)] if kind == "static" else [out, len(rows), info, None]
