"""The work that users of this framework have it do, as cases that can be timed.

Every case goes through the public binding (`paper_2003_01527_gb300.gsm`): a
`Matcher` with a resident data graph, queries, and output buffers are what a
program has in hand (`prepare`); one call of the matcher, or one burst of
requests to its server, is one pass (`run`).

Graphs are of the kinds the repository's own workloads use: Erdos-Renyi and
R-MAT (a=.57 b=.19 c=.19, edge factor 16), with uniform or Zipf vertex labels
or none; queries are named shapes or random walks in the data graph.  On a
power-law graph an unrestricted labelled query has up to 10^18 embeddings, so
listings are root slices, as in the repository's workloads: query vertex 0 is
restricted to a window of ids whose embeddings along the query's spanning
tree number at most `rows` (an upper bound of every level's partial
embeddings; exact for trees without repeated labels).
"""
from __future__ import annotations

import itertools
import math

import numpy as np
import torch

from paper_2003_01527_gb300 import gsm

EDGE_FACTOR = 16
SHAPES = {
    "path3": (3, [(0, 1), (1, 2)]),
    "triangle": (3, [(0, 1), (1, 2), (0, 2)]),
    "cycle4": (4, [(0, 1), (1, 2), (2, 3), (0, 3)]),
    "clique4": (4, [(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3)]),
    "cycle5": (5, [(0, 1), (1, 2), (2, 3), (3, 4), (0, 4)]),
    "path6": (6, [(0, 1), (1, 2), (2, 3), (3, 4), (4, 5)]),
}


def listed():
    return [
        # The smallest call: one labelled 4-cycle in a small Erdos-Renyi graph
        # (2,000 vertices, degree 8, 4 labels), sorted rows back on the host.
        # What an interactive user waits for: launches and read-backs.
        {"name": "tiny_er_list", "op": "list_host", "graph": "er", "n": 2000, "labels": 4,
         "zipf": 0.0, "shape": "cycle4", "queries": 1, "rows": 0},
        # A program that is handed a graph in host memory, loads it and lists
        # one query of it into a pinned host buffer, as in a pipeline over
        # many graphs: upload, load-time tables, one listing, copy back.
        {"name": "load_and_list", "op": "load_list", "graph": "rmat", "scale": 16, "labels": 8,
         "zipf": 1.0, "kmin": 5, "kmax": 5, "extra": -1, "queries": 1, "rows": 1 << 20},
        # The throughput listing: 20 random-walk queries of 4-8 vertices
        # (induced edges) on labelled R-MAT 16, one call, sorted rows on the
        # device.
        {"name": "list_many_rmat16", "op": "list_many", "graph": "rmat", "scale": 16, "labels": 8,
         "zipf": 1.0, "kmin": 4, "kmax": 8, "extra": -1, "queries": 20, "rows": 1 << 23},
        # One large listing of a tree query: the result itself (16 M rows) is
        # the work, and its canonical order.
        {"name": "list_large_rmat16", "op": "list", "graph": "rmat", "scale": 16, "labels": 8,
         "zipf": 1.0, "kmin": 4, "kmax": 4, "extra": 0, "queries": 1, "rows": 1 << 24},
        # Unlabelled listing on a graph larger than L2's reach: a slice of the
        # 5-cycles of R-MAT 20.
        {"name": "list_cycle5_rmat20", "op": "list", "graph": "rmat", "scale": 20, "labels": 1,
         "zipf": 0.0, "shape": "cycle5", "queries": 1, "rows": 1 << 26},
        # A listing whose partial embeddings exceed the memory budget, which
        # forces chunked levels (5-cycles, up to 500 MB of frontiers in 64 MB).
        {"name": "list_cycle5_budget", "op": "list", "graph": "rmat", "scale": 18, "labels": 1,
         "zipf": 0.0, "shape": "cycle5", "queries": 1, "rows": 1 << 25, "budget_mb": 64},
        # Counting without listing, every embedding a candidate: all 2-edge
        # paths of R-MAT 20 (7 x 10^10).
        {"name": "count_path3_rmat20", "op": "count", "graph": "rmat", "scale": 20, "labels": 1,
         "zipf": 0.0, "shape": "path3", "queries": 1, "rows": 0},
        # All ordered triangles of R-MAT 20: the count that verification
        # bounds.
        {"name": "count_triangle_rmat20", "op": "count", "graph": "rmat", "scale": 20, "labels": 1,
         "zipf": 0.0, "shape": "triangle", "queries": 1, "rows": 0},
        # Distinct subgraphs up to automorphism: 4-cliques of R-MAT 16.
        {"name": "distinct_clique4_rmat16", "op": "distinct", "graph": "rmat", "scale": 16,
         "labels": 1, "zipf": 0.0, "shape": "clique4", "queries": 1, "rows": 0},
        # The batched form: 256 uneven queries (3-10 vertices, 2-4 non-tree
        # edges) on labelled R-MAT 18, counted as one batch.
        {"name": "batch_count_rmat18", "op": "batch", "graph": "rmat", "scale": 18, "labels": 16,
         "zipf": 1.2, "kmin": 3, "kmax": 10, "extra": 4, "queries": 256, "rows": 1 << 18},
        # ... and listed: 48 queries, sorted rows on the device.
        {"name": "batch_list_rmat18", "op": "batch_list", "graph": "rmat", "scale": 18,
         "labels": 16, "zipf": 1.2, "kmin": 3, "kmax": 10, "extra": 4, "queries": 48,
         "rows": 1 << 18},
        # The served form: a burst of 48 requests, half counted and half
        # listed, submitted and polled until all are answered.
        {"name": "served_burst_rmat18", "op": "served", "graph": "rmat", "scale": 18, "labels": 32,
         "zipf": 1.0, "kmin": 3, "kmax": 8, "extra": 2, "queries": 48, "rows": 1 << 14},
    ]


def _log_int(rng, lo, hi):
    """A whole number, spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    case = _draw(rng)
    if case["graph"] == "rmat":  # vertex counts that fill no word, other densities
        case["n"] = (1 << case["scale"]) - rng.randint(0, 1 << (case["scale"] - 2))
        case["edge_factor"] = rng.randint(6, EDGE_FACTOR)
    return case


def _draw(rng):
    op = rng.choice(["list_host", "load_list", "list_many", "list", "list", "list_shape", "budget",
                     "count", "count_walk", "distinct", "batch", "batch_list", "served"])
    walk = {"graph": "rmat", "scale": rng.randint(13, 18), "labels": rng.choice([4, 7, 8, 16, 32]),
            "zipf": rng.choice([1.0, 1.2]), "queries": 1}
    k = rng.randint(3, 8)
    if op == "list_host":
        return {"op": op, "graph": "er", "n": _log_int(rng, 300, 20000),
                "labels": rng.choice([1, 2, 4, 5]), "zipf": 0.0,
                "shape": rng.choice(["triangle", "cycle4", "cycle5", "path3"]), "queries": 1,
                "rows": 0}
    if op == "load_list":
        return dict(walk, op=op, kmin=k, kmax=k, extra=-1, rows=_log_int(rng, 1 << 10, 1 << 20))
    if op == "list_many":
        return dict(walk, op=op, kmin=3, kmax=k, extra=rng.choice([-1, 0, 2]),
                    queries=rng.randint(2, 20), rows=_log_int(rng, 1 << 10, 1 << 22))
    if op == "list":
        return dict(walk, op=op, kmin=k, kmax=k, extra=rng.choice([-1, 0, 2]),
                    rows=_log_int(rng, 100, 1 << 24), compressed=rng.random() < 0.25)
    if op == "list_shape":
        return {"op": "list", "graph": "rmat", "scale": rng.randint(14, 20), "labels": 1,
                "zipf": 0.0, "shape": rng.choice(["triangle", "cycle4", "clique4", "cycle5"]),
                "queries": 1, "rows": _log_int(rng, 1 << 12, 1 << 26)}
    if op == "budget":
        return {"op": "list", "graph": "rmat", "scale": rng.randint(14, 18), "labels": 1,
                "zipf": 0.0, "shape": rng.choice(["cycle4", "cycle5"]), "queries": 1,
                "rows": _log_int(rng, 1 << 20, 1 << 25), "budget_mb": rng.choice([32, 48, 64, 96]),
                "compressed": rng.random() < 0.3}
    if op == "count":
        shape = rng.choice(["path3", "triangle", "triangle", "cycle4", "clique4"])
        top = {"path3": 20, "triangle": 20, "cycle4": 12, "clique4": 14}[shape]
        return {"op": op, "graph": "rmat", "scale": rng.randint(12, top), "labels": 1, "zipf": 0.0,
                "shape": shape, "queries": 1, "rows": 0}
    if op == "count_walk":
        return dict(walk, op="count", kmin=k, kmax=k, extra=rng.choice([-1, 0, 2]),
                    rows=_log_int(rng, 1 << 10, 1 << 30))
    if op == "distinct":
        shape = rng.choice(["triangle", "clique4", "cycle4"])
        top = {"triangle": 20, "clique4": 16, "cycle4": 12}[shape]
        return {"op": op, "graph": "rmat", "scale": rng.randint(12, top), "labels": 1, "zipf": 0.0,
                "shape": shape, "queries": 1, "rows": 0}
    if op == "served":
        return dict(walk, op=op, kmin=3, kmax=k, extra=rng.choice([-1, 0, 2]),
                    queries=rng.randint(1, 48), rows=_log_int(rng, 1 << 8, 1 << 14))
    top = 256 if op == "batch" else 48
    return dict(walk, op=op, kmin=3, kmax=rng.randint(k, 10), extra=rng.choice([-1, 2, 4]),
                queries=_log_int(rng, 4, top), rows=_log_int(rng, 1 << 8, 1 << 18))


# ------------------------------------------------------------------ inputs


def _graph(case, seed):
    """(n, row_ptr, col, labels), int32 on the device: sorted symmetric CSR
    without self-loops or duplicates."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    if case["graph"] == "er":
        n, m = case["n"], 4 * case["n"]
        src = torch.randint(0, n, (m,), generator=gen, device="cuda")
        dst = torch.randint(0, n, (m,), generator=gen, device="cuda")
    else:
        n, m = 1 << case["scale"], case.get("edge_factor", EDGE_FACTOR) << case["scale"]
        src = torch.zeros(m, dtype=torch.int64, device="cuda")
        dst = torch.zeros(m, dtype=torch.int64, device="cuda")
        for bit in range(case["scale"]):
            u = torch.rand(m, generator=gen, device="cuda")
            src |= (u >= 0.76).to(torch.int64) << bit
            dst |= (((u >= 0.57) & (u < 0.76)) | (u >= 0.95)).to(torch.int64) << bit
        perm = torch.randperm(n, generator=gen, device="cuda")
        src, dst = perm[src], perm[dst]
        n = case.get("n", n)
    keep = (src != dst) & (src < n) & (dst < n)
    src, dst = src[keep], dst[keep]
    keys = torch.unique(torch.cat([src * n + dst, dst * n + src]))
    col = (keys % n).to(torch.int32)
    deg = torch.bincount(torch.div(keys, n, rounding_mode="floor"), minlength=n)
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(deg, 0, out=rp[1:])
    L = case["labels"]
    p = (torch.arange(1, L + 1, dtype=torch.float64) ** -case["zipf"]).cuda()
    u = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
    lab = torch.searchsorted(torch.cumsum(p / p.sum(), 0), u).clamp(max=L - 1)
    return n, rp.to(torch.int32), col, lab.to(torch.int32)


def _walk_query(rp, col, lab, k, extra, rng):
    """A connected query cut out of the graph by a random walk: its
    first-visit tree edges, plus every other induced edge (extra < 0) or at
    most `extra` of them."""
    best = None
    for _ in range(1 if extra <= 0 else 6):
        while True:
            cur = int(rng.integers(0, len(rp) - 1))
            if rp[cur + 1] == rp[cur]:
                continue
            seen, tree = [cur], []
            for _ in range(50 * k):
                nxt = int(col[rng.integers(rp[cur], rp[cur + 1])])
                if nxt not in seen:
                    tree.append((seen.index(cur), len(seen)))
                    seen.append(nxt)
                    if len(seen) == k:
                        break
                cur = nxt
            if len(seen) == k:
                break
        more = []
        for a in range(k if extra else 0):
            row = col[rp[seen[a]]:rp[seen[a] + 1]]
            for b in range(a + 1, k):
                at = np.searchsorted(row, seen[b])
                if at < len(row) and row[at] == seen[b] and (a, b) not in tree:
                    more.append((a, b))
        if extra > 0 and len(more) > extra:
            more = [more[i] for i in sorted(rng.choice(len(more), extra, replace=False))]
        if best is None or len(more) > len(best[1]):
            best = (seen, more, tree)
        if extra < 0 or len(more) >= extra:
            break
    seen, more, tree = best
    return k, sorted(tree + more), [int(lab[v]) for v in seen], seen[0]


def _order(k, edges, sizes):
    """Connected matching order from query vertex 0 and each position's tree
    parent: most edges to placed vertices, then fewest candidates."""
    adj = [{b for a, b in edges if a == u} | {a for a, b in edges if b == u} for u in range(k)]
    order = [0]
    while len(order) < k:
        rest = [u for u in range(k) if u not in order and adj[u] & set(order)]
        order.append(min(rest, key=lambda u: (-len(adj[u] & set(order)), sizes[u], -len(adj[u]), u)))
    return adj, order, [None] + [next(p for p in order if p in adj[u]) for u in order[1:]]


def _window(graph, query, start, rows):
    """The ids [lo, hi) for query vertex 0 with the most spanning-tree
    embeddings among the windows of at most `rows` of them (dead ends count
    too), and with fewer root candidates than any other query vertex has; a
    window that holds `start` (the walk's own root) if there is one."""
    n, rp, col, lab = graph
    k, edges, qlab = query
    rp = rp.to(torch.int64)
    deg = rp[1:] - rp[:-1]
    qdeg = [sum(u in e for e in edges) for u in range(k)]
    cand = [(lab == qlab[u]) & (deg >= qdeg[u]) for u in range(k)]
    sizes = [int(x) for x in torch.stack([c.sum() for c in cand]).tolist()]
    _, order, parent = _order(k, edges, sizes)
    top = float(1 << 40)
    h = [c.to(torch.int64) for c in cand]
    csum = torch.zeros(col.numel() + 1, dtype=torch.int64, device="cuda")
    at = col.to(torch.int64)
    for u, p in reversed(list(zip(order[1:], parent[1:]))):
        torch.cumsum(h[u][at], 0, out=csum[1:])
        s = (csum[rp[1:]] - csum[rp[:-1]]).clamp(min=1)
        h[p] = (h[p].to(torch.float64) * s.to(torch.float64)).clamp(max=top).to(torch.int64)
    cs = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(h[0], 0, out=cs[1:])
    roots = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    torch.cumsum(cand[0], 0, out=roots[1:])
    end = torch.searchsorted(cs, cs + rows, right=True) - 1
    most = max(1, min(sizes[1:]) - 1)
    end = torch.minimum(end, torch.searchsorted(roots, roots + most, right=True) - 1)
    value = cs[end] - cs
    if start >= 0:
        ids = torch.arange(n + 1, device="cuda")
        held = (ids <= start) & (end > start)
        if bool(held.any()):
            value = torch.where(held, value, torch.zeros_like(value))
        else:
            start = -1
    lo = int((value == value.max()).nonzero()[0, 0])
    return lo, max(lo, int(end[lo])), start >= 0


def _sizes(case):
    """The query sizes of a case: spread over kmin..kmax, the same for every
    seed."""
    span = case["kmax"] - case["kmin"] + 1
    return [case["kmin"] + (5 * j + 2) % span for j in range(case["queries"])]


def _inputs(case, seed):
    """The graph and its queries: [(k, edges, labels, lo, hi)]."""
    graph = _graph(case, seed)
    n, rp, col, lab = graph
    rng = np.random.default_rng(seed)
    queries = []
    if "shape" in case:
        k, edges = SHAPES[case["shape"]]
        qlab = [(0, 1, 0, 2, 1)[u] % case["labels"] for u in range(k)]
        window = _window(graph, (k, edges, qlab), -1, case["rows"]) if case["rows"] else (0, n)
        queries.append((k, edges, qlab) + window[:2])
    else:
        h_rp, h_col, h_lab = rp.cpu().numpy(), col.cpu().numpy(), lab.cpu().numpy()
        for k in _sizes(case):
            # a walk whose own embedding lies in the slice, if a few tries
            # find one (hub-heavy walks have more than `rows` embeddings)
            for _ in range(32 if case["queries"] == 1 else 4):
                *query, start = _walk_query(h_rp, h_col, h_lab, k, case["extra"], rng)
                lo, hi, holds = _window(graph, query, start, case["rows"])
                if holds:
                    break
            queries.append((*query, lo, hi))
    torch.cuda.synchronize()
    return graph, queries


def _room(case, k):
    """Rows of the buffer that a program keeps for one query's result."""
    if case["rows"]:
        return case["rows"]
    return 100 * case["n"] if case["shape"] == "path3" else 2 * 8 ** k + 1024


def prepare(case, seed):
    graph, queries = _inputs(case, seed)
    n, rp, col, lab = graph
    op = case["op"]
    m = gsm.Matcher(device=0, mem_budget_bytes=case.get("budget_mb", 0) << 20,
                    compressed=case.get("compressed", False))
    state = {"op": op, "matcher": m, "queries": []}
    for k, edges, qlab, lo, hi in queries:
        q = m.query(k, edges, qlab)
        if case["rows"]:
            q.restrict(0, lo, hi)
        state["queries"].append(q)
    ints = [k * _room(case, k) for k, *_ in queries] if op not in ("count", "distinct", "batch") else []
    if op == "load_list":
        state["graph"] = [t.cpu().numpy() for t in (rp, col, lab)]
        state["out"] = torch.zeros(ints[0], dtype=torch.int32).pin_memory()
        return state
    m.load_graph(rp, col, lab if case["labels"] > 1 else None)
    if op in ("list", "list_many"):
        state["outs"] = [torch.zeros(i, dtype=torch.int32, device="cuda") for i in ints]
    elif op == "batch_list":
        state["out"] = torch.zeros(sum(ints), dtype=torch.int32, device="cuda")
    elif op == "list_host":
        state["out"] = np.zeros(ints[0], dtype=np.int32)
    elif op == "served":
        state["out"] = np.zeros(sum(ints[1::2]), dtype=np.int32)
        gsm.gsm_server_start(m.ctx, 2, 64)
    torch.cuda.synchronize()
    return state


def _keep(out, rows):
    """Puts the results a call handed out into the program's own buffer, one
    after the other."""
    flat = [r.reshape(-1) for r in rows]
    total = sum(len(r) for r in flat)
    if isinstance(out, np.ndarray):
        np.concatenate(flat, out=out[:total])
    else:
        torch.cat(flat, out=out[:total])
    return out


def run(state):
    op, m, qs = state["op"], state["matcher"], state["queries"]
    if op == "list_host":
        rows, count = m.enumerate(qs[0])
        return {"rows": _keep(state["out"], [rows]), "count": count}
    if op == "load_list":
        m.load_graph(*state["graph"])
        out, count = m.enumerate(qs[0], out=state["out"])
        return {"rows": out, "count": count}
    if op == "list":
        out, count = m.enumerate(qs[0], out=state["outs"][0])
        return {"rows": out, "count": count}
    if op == "list_many":
        counts = m.enumerate_many(qs, state["outs"])
        return {"rows": state["outs"], "counts": np.array(counts, dtype=np.int64)}
    if op == "count":
        return {"count": m.count(qs[0])}
    if op == "distinct":
        count, automorphisms = m.count_distinct(qs[0])
        return {"count": count, "automorphisms": automorphisms}
    if op == "batch":
        return {"counts": np.array(m.run_batch(qs), dtype=np.int64)}
    if op == "batch_list":
        counts, rows = m.run_batch(qs, enumerate=True, device=True)
        return {"rows": _keep(state["out"], rows), "counts": np.array(counts, dtype=np.int64)}
    tickets = [gsm.gsm_submit(m.ctx, q.handle, gsm.GSM_MODE_ENUMERATE if j % 2 else gsm.GSM_MODE_COUNT)
               for j, q in enumerate(qs)]
    done = [None] * len(tickets)
    while any(d is None for d in done):
        for j, t in enumerate(tickets):
            if done[j] is None:
                done[j] = gsm.gsm_poll(m.ctx, t)
    rows = [d["rows"] for d in done if "rows" in d]
    return {"rows": _keep(state["out"], rows) if rows else state["out"],
            "counts": np.array([d["count"] for d in done], dtype=np.int64)}


def work(case):
    """One read of the graph and one write of the result (for slices, its
    bound: the rows of a tree query, more than a query with cycles has); the
    served and batched forms read the graph once for all their queries."""
    if case["graph"] == "er":
        n, nnz = case["n"], 8 * case["n"]
    else:
        n = case.get("n", 1 << case["scale"])
        nnz = int(2 * case.get("edge_factor", EDGE_FACTOR) * n * 0.9)
    labels = 4 * n if case["labels"] > 1 else 0
    size = 4 * (n + 1) + 4 * nnz + labels
    if case["op"] in ("list", "list_many", "load_list", "batch_list"):
        k = SHAPES[case["shape"]][0] if "shape" in case else (case["kmin"] + case["kmax"]) / 2
        share = 1.0 if case.get("extra") == 0 else 0.1
        size += 4 * k * case["rows"] * case["queries"] * share
    return {"bytes": size, "flops": 0}


# ------------------------------------------------------------------ exact

_MOST = 1 << 27  # candidates of one level that exact() takes on


def _automorphisms(k, edges, labels):
    es = {frozenset(e) for e in edges}
    return sum(all(labels[p[u]] == labels[u] for u in range(k)) and
               {frozenset((p[a], p[b])) for a, b in edges} == es
               for p in itertools.permutations(range(k)))


def _join(graph, query):
    """Sorted embeddings of one query by joins over the edge list (int64), or
    None where a level has more than _MOST candidates."""
    n, rp, col, lab = graph
    k, edges, qlab, lo, hi = query
    rp, col = rp.to(torch.int64), col.to(torch.int64)
    deg = rp[1:] - rp[:-1]
    keys = torch.repeat_interleave(torch.arange(n, device="cuda"), deg) * n + col
    sizes = torch.bincount(lab, minlength=max(qlab) + 1).tolist()
    adj, order, parent = _order(k, edges, [sizes[l] for l in qlab])
    root = torch.arange(lo, min(hi, n), device="cuda")
    rows = root[(lab[root] == qlab[0]) & (deg[root] >= len(adj[0]))][:, None]
    for i in range(1, k):
        u = order[i]
        x = rows[:, order.index(parent[i])]
        d = deg[x]
        total = int(d.sum())
        if total > _MOST:
            return None
        r = torch.repeat_interleave(torch.arange(len(x), device="cuda"), d)
        first = torch.cumsum(d, 0) - d
        w = col[rp[x][r] + torch.arange(total, device="cuda") - first[r]]
        ok = lab[w] == qlab[u]
        r, w = r[ok], w[ok]
        ok = deg[w] >= len(adj[u])
        for j in range(i):
            y = rows[r, j]
            ok &= y != w
            if order[j] in adj[u] and order[j] != parent[i] and keys.numel():
                key = y * n + w
                at = torch.searchsorted(keys, key).clamp(max=keys.numel() - 1)
                ok &= keys[at] == key
        rows = torch.cat([rows[r[ok]], w[ok][:, None]], 1)
    rows = rows[:, [order.index(u) for u in range(k)]]
    for c in range(k - 1, -1, -1):
        rows = rows[torch.sort(rows[:, c], stable=True)[1]]
    return rows


def _cliques(graph, k):
    """Distinct k-cliques (k = 3, 4): edges oriented along increasing degree,
    wedges joined in pieces."""
    n, rp, col, _ = graph
    rp, col = rp.to(torch.int64), col.to(torch.int64)
    deg = rp[1:] - rp[:-1]
    rank = torch.empty_like(deg)
    rank[torch.sort(deg, stable=True)[1]] = torch.arange(n, device="cuda")
    a, b = rank[torch.repeat_interleave(torch.arange(n, device="cuda"), deg)], rank[col]
    keys = torch.sort((a * n + b)[a < b])[0]
    if not keys.numel():
        return 0
    b = keys % n
    out = torch.bincount(torch.div(keys, n, rounding_mode="floor"), minlength=n)
    first = torch.cumsum(out, 0) - out

    def has(x, y):
        at = torch.searchsorted(keys, x * n + y).clamp(max=keys.numel() - 1)
        return keys[at] == x * n + y

    def grow(rows, last):
        """The number of cliques that extend the rows (ranks increasing)."""
        d = out[rows[:, -1]]
        ends = torch.cumsum(d, 0)
        total, done, lo = 0, 0, 0
        while lo < len(rows):
            hi = max(lo + 1, int(torch.searchsorted(ends, done + (_MOST >> 2), right=True)))
            piece, dd = rows[lo:hi], d[lo:hi]
            r = torch.repeat_interleave(torch.arange(len(piece), device="cuda"), dd)
            at = torch.arange(len(r), device="cuda") - (torch.cumsum(dd, 0) - dd)[r]
            w = b[first[piece[:, -1]][r] + at]
            ok = torch.ones_like(w, dtype=torch.bool)
            for c in range(rows.shape[1] - 1):
                ok &= has(piece[r, c], w)
            if last:
                total += int(ok.sum())
            else:
                total += grow(torch.cat([piece[r[ok]], w[ok][:, None]], 1), True)
            done, lo = int(ends[hi - 1]), hi
        return total

    edges = torch.stack([torch.div(keys, n, rounding_mode="floor"), b], 1)
    return grow(edges, k == 3)


def exact(case, seed):
    graph, queries = _inputs(case, seed)
    op = case["op"]
    if op in ("count", "distinct") and not case["rows"]:
        k, edges, qlab = queries[0][:3]
        aut = _automorphisms(k, edges, qlab)
        if case["shape"] == "path3":
            d = (graph[1][1:] - graph[1][:-1]).to(torch.int64)
            count = int((d * (d - 1)).sum())
        elif case["shape"] in ("triangle", "clique4") and case["scale"] <= (20 if k == 3 else 16):
            count = _cliques(graph, k) * aut
        else:
            return None
        return {"count": count} if op == "count" else {"count": count // aut, "automorphisms": aut}
    rows = [_join(graph, q) for q in queries]
    if any(r is None for r in rows):
        return None
    counts = np.array([len(r) for r in rows], dtype=np.int64)
    if op == "count":
        return {"count": int(counts[0])}
    if op == "batch":
        return {"counts": counts}

    def laid(some):
        """The rows one after the other in a buffer of their queries' room."""
        out = torch.zeros(sum(r.shape[1] * _room(case, r.shape[1]) for r in some), dtype=torch.int32)
        flat = torch.cat([r.reshape(-1) for r in some]) if some else torch.zeros(0)
        out[:len(flat)] = flat.to(torch.int32).cpu()
        return out

    if op == "list_many":
        return {"rows": [laid([r]) for r in rows], "counts": counts}
    if op in ("batch_list", "served"):
        return {"rows": laid(rows[1::2] if op == "served" else rows), "counts": counts}
    return {"rows": laid(rows), "count": int(counts[0])}
