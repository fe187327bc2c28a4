"""gsm_count's shortcuts against the oracle: queries whose leaves are
multiplied out instead of extended (one and several parents, equal and
different labels, restricted leaves), queries with symmetries (one of every
set of symmetric embeddings is counted; candidates outside the ordering
constraints are never generated), and counts past 64 bits."""
import math
import time

import numpy as np
import pytest

import oracle
from paper_2003_01527_gb300 import inputs as I

pytestmark = pytest.mark.gpu

SHAPES = {
    "edge": (2, [(0, 1)]),
    "path3": (3, [(0, 1), (1, 2)]),
    "path5": (5, [(0, 1), (1, 2), (2, 3), (3, 4)]),
    "star5": (6, [(0, 1), (0, 2), (0, 3), (0, 4), (0, 5)]),
    "tailed_triangle": (5, [(0, 1), (1, 2), (0, 2), (2, 3), (3, 4)]),
    "bull": (5, [(0, 1), (1, 2), (0, 2), (0, 3), (1, 4)]),
    "triangle_two_tails": (5, [(0, 1), (1, 2), (0, 2), (2, 3), (2, 4)]),
    "caterpillar": (7, [(0, 1), (1, 2), (0, 3), (1, 4), (1, 5), (2, 6)]),
    "triangle": (3, [(0, 1), (1, 2), (0, 2)]),
    "cycle4": (4, [(0, 1), (1, 2), (2, 3), (0, 3)]),
    "diamond": (4, [(0, 1), (1, 2), (2, 3), (0, 3), (0, 2)]),
    "clique4": (4, [(0, 1), (0, 2), (0, 3), (1, 2), (1, 3), (2, 3)]),
    "cycle5": (5, [(0, 1), (1, 2), (2, 3), (3, 4), (0, 4)]),
    "k23": (5, [(0, 2), (0, 3), (0, 4), (1, 2), (1, 3), (1, 4)]),
    "cycle6": (6, [(0, 1), (1, 2), (2, 3), (3, 4), (4, 5), (0, 5)]),
    "square_with_tails": (6, [(0, 1), (1, 2), (2, 3), (0, 3), (0, 4), (2, 5)]),
}


def er(n, m, labels, seed):
    _, rp, col = I.erdos_renyi(n, m, seed=seed)
    lab = I.uniform_labels(n, labels, seed + 1) if labels > 1 else np.zeros(n, np.int32)
    return I.make_graph(n, rp, col, lab)


@pytest.mark.parametrize("labels", [1, 2, 3])
@pytest.mark.parametrize("shape", sorted(SHAPES))
def test_counts_of_shapes(gsm_lib, cuda, shape, labels):
    g = er(90, 500, labels, seed=50 + labels)
    k, edges = SHAPES[shape]
    rng = np.random.default_rng(labels)
    m = gsm_lib.Matcher(device=0)
    m.load_graph(g.row_ptr, g.col, g.labels, validate=True)
    others = [gsm_lib.Matcher(device=0, **o) for o in
              ({"mem_budget_bytes": 1 << 18, "chunk_rows": 37}, {"compressed": True},
               {"lookahead": 2}, {"two_pass": True, "hub_bitmap_bytes": -1, "filter_rounds": 1})]
    for x in others:
        x.load_graph(g.row_ptr, g.col, g.labels)
    for trial in range(4 if labels > 1 else 1):
        q = I.query_from_edges(k, edges, rng.integers(0, labels, k))
        want = oracle.count(g, q)
        for x in [m] + others:
            assert x.count(x.query(q.k, q.edges, q.labels)) == want
        distinct, aut = m.count_distinct(m.query(q.k, q.edges, q.labels))
        assert distinct * aut == want
        # a range of every vertex in turn: results of the two parts add up
        for u in range(k):
            parts = [m.count(m.query(q.k, q.edges, q.labels).restrict(u, *r))
                     for r in ((0, 31), (31, g.n))]
            assert sum(parts) == want
        # every vertex restricted, alike and each to its own range: the count
        # and the listing are the rows of the whole result in the ranges
        rows = oracle.match(g, q)[1]
        for ranges in ([(7, 70)] * k, [(5, 60 + 3 * u) for u in range(k)]):
            keep = np.all([(rows[:, u] >= a) & (rows[:, u] < b)
                           for u, (a, b) in enumerate(ranges)], axis=0)
            for x in [m] + others:
                Q = x.query(q.k, q.edges, q.labels)
                for u, r in enumerate(ranges):
                    Q.restrict(u, *r)
                assert x.count(Q) == int(keep.sum())
                assert np.array_equal(x.enumerate(Q)[0], rows[keep])
    for x in [m] + others:
        x.close()


def test_counts_past_64_bits(gsm_lib, cuda):
    """A star with d leaves has perm(d, m) maps of an m-leaf star onto its
    centre (m >= 2): exact below 2^64, an error above."""
    d = 2000
    g = I.graph_from_edges(d + 1, [(0, v) for v in range(1, d + 1)])
    m = gsm_lib.Matcher(device=0)
    m.load_graph(g.row_ptr, g.col, g.labels)

    def star(leaves):
        return m.query(leaves + 1, [(0, j + 1) for j in range(leaves)])

    assert math.perm(d, 5) < 2 ** 64 < math.perm(d, 6)
    assert m.count(star(5)) == math.perm(d, 5)
    for leaves in (6, 9, 15):
        with pytest.raises(gsm_lib.GsmError) as e:
            m.count(star(leaves))
        assert e.value.status == gsm_lib.GSM_ERR_OVERFLOW
    assert m.count(star(3)) == math.perm(d, 3)  # the context is still usable
    # 40 hubs of 2,000 leaves: every hub's number fits in 64 bits, and their sum
    hubs = I.graph_from_edges(40 * 2001, [(2001 * h, 2001 * h + v) for h in range(40)
                                          for v in range(1, 2001)])
    m.load_graph(hubs.row_ptr, hubs.col, hubs.labels)
    assert m.count(star(4)) == 40 * math.perm(2000, 4)
    with pytest.raises(gsm_lib.GsmError) as e:
        m.count(star(6))
    assert e.value.status == gsm_lib.GSM_ERR_OVERFLOW
    m.close()


def test_one_count_past_64_bits_is_not_the_others(gsm_lib, cuda):
    """A batch with a count past 64 bits reports it, with every other count;
    in the served form only that request fails, listings beside it too."""
    d = 2000
    g = I.graph_from_edges(d + 4, [(0, v) for v in range(1, d + 1)] +
                           [(d + 1, d + 2), (d + 2, d + 3), (d + 1, d + 3)])
    m = gsm_lib.Matcher(device=0)
    m.load_graph(g.row_ptr, g.col, g.labels)
    star = [m.query(x + 1, [(0, j + 1) for j in range(x)]) for x in range(1, 9)]
    triangle = m.query(3, [(0, 1), (1, 2), (0, 2)])
    want = [math.perm(d, x) + (6 if x < 3 else 0) for x in range(1, 9)] + [6]
    want[0] = 2 * (d + 3)
    capped = [min(c, 2 ** 64 - 1) for c in want]
    assert capped.count(2 ** 64 - 1) == 3
    for _ in range(2):
        with pytest.raises(gsm_lib.GsmError) as e:
            m.run_batch(star + [triangle])
        assert e.value.status == gsm_lib.GSM_ERR_OVERFLOW
        assert [int(c) for c in e.value.counts] == capped
    assert m.run_batch(star[:5] + [triangle]) == want[:5] + [6]
    tri = [[d + 1 + a, d + 1 + b, d + 1 + c] for a, b, c in
           [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]]
    gsm_lib.gsm_server_start(m.ctx, 2, 16)
    tickets = [gsm_lib.gsm_submit(m.ctx, q.handle) for q in star]
    tickets.append(gsm_lib.gsm_submit(m.ctx, triangle.handle, gsm_lib.GSM_MODE_ENUMERATE))
    done = [None] * len(tickets)
    deadline = time.time() + 60
    while None in done and time.time() < deadline:
        done = [r or gsm_lib.gsm_poll(m.ctx, t) for r, t in zip(done, tickets)]
    gsm_lib.gsm_server_stop(m.ctx)
    assert None not in done
    for r, c in zip(done, want):
        if c < 2 ** 64:
            assert (r["status"], r["count"]) == (gsm_lib.GSM_OK, c)
        else:
            assert r["status"] == gsm_lib.GSM_ERR_OVERFLOW
    assert done[-1]["rows"].tolist() == tri
    m.close()


def test_sums_of_halves_past_64_bits(gsm_lib, cuda):
    """In K_n, a vertex with three leaves and a tail of two has n (n-1) (n-2)
    core embeddings, each with (n-3) (n-4) (n-5) images of the leaves.  At n =
    1,629 that is more than 2^32 embeddings of just under 2^32 each: their
    numbers' low halves add up past 64 bits, the high ones to nothing."""
    edges = [(0, 1), (0, 2), (0, 3), (0, 4), (4, 5)]
    m = gsm_lib.Matcher(device=0)
    for n in (1626, 1629):
        ids = np.arange(n * n, dtype=np.int64)
        src, dst = ids // n, ids % n
        rp, col = I.csr_from_pairs(n, src[src != dst], dst[src != dst])
        m.load_graph(rp, col)
        assert n * (n - 1) * (n - 2) > 2 ** 32 - 2 ** 28
        assert (n - 3) * (n - 4) * (n - 5) < 2 ** 32
        want = math.perm(n, 6)
        if want < 2 ** 64:
            assert m.count(m.query(6, edges)) == want
            continue
        with pytest.raises(gsm_lib.GsmError) as e:
            m.count(m.query(6, edges))
        assert e.value.status == gsm_lib.GSM_ERR_OVERFLOW
    m.close()


@pytest.mark.parametrize("hub_bytes", [0, -1, 1 << 16])
def test_cliques_on_the_renumbered_graph(gsm_lib, cuda, hub_bytes):
    """Unrestricted cliques on a one-label graph with enough 2-edge paths are
    counted with its vertices renumbered by degree; a partition into root
    ranges (never renumbered) adds up to the same, and the first one loaded
    afterwards does not see the old numbering."""
    m = gsm_lib.Matcher(device=0, hub_bitmap_bytes=hub_bytes)
    for scale, ef, drop in ((15, 16, 77), (14, 40, 3)):
        n, rp, col = I.rmat(scale, ef, *I.RMAT_ABC, seed=91)
        src = np.repeat(np.arange(n), np.diff(rp))
        keep = (src < n - drop) & (col < n - drop)  # vertices that fill no bitmap word
        n -= drop
        rp, col = I.csr_from_pairs(n, src[keep], col[keep])
        d = np.diff(rp).astype(float)
        assert (d * d).sum() > 2 ** 28
        m.load_graph(rp, col, validate=True)
        for k in (3, 4, 5):
            edges = [(i, j) for i in range(k) for j in range(i + 1, k)]
            if k == 5 and scale == 14:
                continue  # the partition takes long
            parts = [m.count(m.query(k, edges).restrict(0, *r))
                     for r in ((0, n // 3), (n // 3, n - 1), (n - 1, n))]
            assert m.count(m.query(k, edges)) == sum(parts), (scale, k)
            assert m.count_distinct(m.query(k, edges)) == \
                (sum(parts) // math.factorial(k), math.factorial(k))
    m.close()


@pytest.mark.parametrize("opts", [{}, {"two_pass": True}, {"compressed": True},
                                  {"block_size": 1024}, {"lookahead": 1}])
def test_long_runs_of_rows_without_candidates(gsm_lib, cuda, opts):
    """A range on the last vertex leaves most rows of a level without
    candidates, in runs longer than a tile's rows, with single rows and short
    gaps between them."""
    n, spokes = 6010, 6000
    pairs = [(0, a) for a in range(1, spokes + 1)]
    for z, at in ((6001, [1, 2, 4, 9, 15, 2500]), (6002, [3, 2501, 2507, 6000]), (6003, [5999]),
                  (6004, [1, 6000])):
        pairs += [(z, a) for a in at] + [(0, z)]
    g = I.graph_from_edges(n, pairs)
    m = gsm_lib.Matcher(device=0, **opts)
    m.load_graph(g.row_ptr, g.col, g.labels)
    windows = [(1, (6001, 6005)), (2, (6001, 6005)), (2, (6003, 6010))]
    for shape in ("path3", "triangle", "cycle4", "diamond"):
        k, edges = SHAPES[shape]
        q = I.query_from_edges(k, edges)
        for u, (lo, hi) in windows:
            ranges = {v: (0, 1) for v in [0] if shape != "diamond"}
            ranges[u] = (lo, hi)
            want, rows, rc = oracle.match(g, q, root_range=ranges.get(0, (0, n)),
                                          ranges={u: (lo, hi)})
            assert rc == oracle.OK
            Q = m.query(k, edges)
            for v, r in ranges.items():
                Q.restrict(v, *r)
            assert m.count(Q) == want, (shape, u)
            got, count = m.enumerate(Q)
            assert count == want and np.array_equal(got, rows), (shape, u)
            if not opts:
                assert m.run_batch([Q, Q]) == [want, want]
    m.close()


@pytest.mark.parametrize("opts", [{}, {"lookahead": 1}, {"block_size": 128}, {"block_size": 512},
                                  {"block_size": 1024, "lookahead": 2}, {"two_pass": True},
                                  {"compressed": True}, {"count_probes": True},
                                  {"hub_bitmap_bytes": -1}])
def test_checks_of_many_neighbours(gsm_lib, cuda, opts):
    """More than three mapped neighbours, with many candidates a row (a dense
    graph) and few (a sparse one with cliques in it), counted and listed, with
    and without a leaf."""
    rng = np.random.default_rng(23)
    cliques = [(int(a), int(b)) for _ in range(30)
               for c in [np.sort(rng.choice(600, 7, replace=False))]
               for i, a in enumerate(c) for b in c[i + 1:]]
    sparse = sorted(set(cliques + [(u, u + 1) for u in range(599)]))
    n, rp, col = I.erdos_renyi(70, 1500, seed=29)
    k5 = [(a, b) for a in range(5) for b in range(a + 1, 5)]
    wheel = [(0, i) for i in range(1, 6)] + [(1, 2), (2, 3), (3, 4), (4, 5), (1, 5)]
    shapes = [(5, k5), (6, wheel), (6, k5 + [(4, 5)]),
              (6, [(a, b) for a in range(6) for b in range(a + 1, 6)])]
    m = gsm_lib.Matcher(device=0, **opts)
    for g in (I.make_graph(n, rp, col, np.arange(n, dtype=np.int32) % 3),
              I.graph_from_edges(600, sparse, np.arange(600, dtype=np.int32) % 2)):
        m.load_graph(g.row_ptr, g.col, g.labels)
        for k, edges in shapes:
            q = I.query_from_edges(k, edges, np.arange(k) % (int(g.labels.max()) + 1))
            hi = 24 if g.n == n else g.n
            want, rows, rc = oracle.match(g, q, root_range=(0, hi))
            assert rc == oracle.OK and want > 0
            Q = m.query(q.k, q.edges, q.labels).restrict(0, 0, hi)
            assert m.count(Q) == want, (k, len(edges))
            got, count = m.enumerate(Q)
            assert count == want and np.array_equal(got, rows), (k, len(edges))
    m.close()
