"""Candidate sets from the graph's threshold bitmaps against the oracle's
filter: requirements at, below and above the bitmaps' four levels, with one
and several labels, vertex counts around a bitmap word, and restrictions that
end inside a word."""
import numpy as np
import pytest

import oracle
from paper_2003_01527_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def graph(n, labels, seed):
    _, rp, col = I.erdos_renyi(n, min(6 * n, n * (n - 1) // 2), seed=seed)
    lab = I.uniform_labels(n, labels, seed + 1) if labels > 1 else np.zeros(n, np.int32)
    return I.make_graph(n, rp, col, lab)


@pytest.mark.parametrize("labels", [1, 2, 5, 70])  # 70: no bitmaps, the row scans
@pytest.mark.parametrize("n", [31, 32, 33, 257, 5000])
def test_candidates_of_stars(gsm_lib, cuda, n, labels):
    g = graph(n, labels, seed=n + labels)
    m = gsm_lib.Matcher(device=0)
    m.load_graph(g.row_ptr, g.col, g.labels, validate=True)
    rng = np.random.default_rng(n)
    for leaves in (1, 3, 4, 5, 8, 12):
        qlab = rng.integers(0, min(labels, 2), leaves + 1)
        q = I.query_from_edges(leaves + 1, [(0, j + 1) for j in range(leaves)], qlab)
        want = np.asarray(oracle.candidates(g, q)).astype(bool)
        for lo, hi in ((0, n), (1, n - 1), (n // 3, n // 2), (32, 64), (n, n + 5)):
            Q = m.query(q.k, q.edges, q.labels).restrict(0, lo, hi)
            bm, sizes = m.candidates(Q)
            got = gsm_lib.unpack_bitmaps(bm, n).astype(bool)
            inside = (np.arange(n) >= lo) & (np.arange(n) < hi)
            assert np.array_equal(got[0], want[0] & inside), (leaves, lo, hi)
            assert np.array_equal(got[1:], want[1:])
            assert [int(s) for s in sizes] == [int(r.sum()) for r in got]
            # no bit past the last vertex
            assert int(np.unpackbits(bm.view(np.uint8)).sum()) == int(got.sum())
    m.close()


@pytest.mark.parametrize("labels", [2, 64, 65])  # 65: sorted, not partitioned row by row
def test_label_segments_of_rows(gsm_lib, cuda, labels):
    """Rows of every length around a warp, the longest row a warp takes (1,024)
    and beyond, some with one label only: the edges between two labels, listed
    through the segments, are numpy's."""
    degrees = [0, 1, 31, 32, 33, 63, 257, 1023, 1024, 1025, 1056, 3001]
    n = len(degrees) + max(degrees)
    rng = np.random.default_rng(labels)
    edges = []
    for h, d in enumerate(degrees):
        ends = len(degrees) + rng.permutation(max(degrees))[:d]
        edges += [(h, int(v)) for v in ends]
    lab = rng.integers(0, labels, n).astype(np.int32)
    lab[len(degrees):len(degrees) + 1200] = 1
    g = I.graph_from_edges(n, edges, lab)
    m = gsm_lib.Matcher(device=0)
    m.load_graph(g.row_ptr, g.col, g.labels, validate=True)
    src = np.repeat(np.arange(n), np.diff(g.row_ptr))
    for a, b in [(0, 1), (1, 0), (1, 1), (int(lab[0]), int(lab[11])), (labels - 1, 1)]:
        keep = (g.labels[src] == a) & (g.labels[g.col] == b)
        want = np.stack([src[keep], g.col[keep]], axis=1)
        rows, count = m.enumerate(m.query(2, [(0, 1)], [a, b]))
        assert count == len(want) and np.array_equal(rows, want), (a, b)
    m.close()
