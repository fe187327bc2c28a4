"""Listings into device memory: what is written there, and until when."""
import numpy as np
import pytest
import torch

import oracle
from paper_2003_01527_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def stars(degrees, pairs=0):
    """One star of label 0 per degree, centres first (ids 0, 1, ...), and
    `pairs` edges between vertices of label 1."""
    c = len(degrees)
    first = np.concatenate([[c], c + np.cumsum(degrees)])
    n = int(first[-1]) + 2 * pairs
    src = np.repeat(np.arange(c), degrees)
    dst = np.arange(c, first[-1])
    a = np.arange(first[-1], n, 2)
    src, dst = np.concatenate([src, a]), np.concatenate([dst, a + 1])
    rp, col = I.csr_from_pairs(n, np.concatenate([src, dst]), np.concatenate([dst, src]))
    lab = (np.arange(n) >= first[-1]).astype(np.int32)
    return I.make_graph(n, rp, col, lab)


@pytest.mark.parametrize("workers", [1, 2])
def test_nothing_is_written_after_a_failed_call_of_many(gsm_lib, cuda, workers):
    """The last query's candidate list does not fit the budget, which the host
    notices without waiting, while the sort of an earlier query's 64 M rows is
    still running: the call waits for it before it returns."""
    d = 8000
    g = stars([d], pairs=1 << 20)
    m = gsm_lib.Matcher(device=0, mem_budget_bytes=4 << 20, host_workers=workers)
    m.load_graph(g.row_ptr, g.col, g.labels)
    path = m.query(3, [(0, 1), (1, 2)], [0, 0, 0])
    edge = m.query(2, [(0, 1)], [1, 1])
    out = torch.empty(3 * d * (d - 1), dtype=torch.int32, device="cuda")
    other = torch.empty(2, dtype=torch.int32, device="cuda")
    assert m.enumerate(path, out=out)[1] == d * (d - 1)  # (buffers have grown)
    for _ in range(2):
        with pytest.raises(gsm_lib.GsmError) as e:
            m.enumerate_many([path, edge, edge], [out, other, other])
        out.fill_(-7)
        torch.cuda.synchronize()
        assert e.value.status == gsm_lib.GSM_ERR_BUDGET
        assert bool((out == -7).all())
    assert m.enumerate_many([path], [out]) == [d * (d - 1)]
    assert out[:6].tolist() == [1, 0, 2, 1, 0, 3]
    m.close()


def test_nothing_is_written_after_a_failed_listing(gsm_lib, cuda):
    """The rows of the first root are being written when the second root's
    partial results turn out not to fit the budget."""
    d = 8000
    g = stars([d, 1 << 20])
    m = gsm_lib.Matcher(device=0, mem_budget_bytes=4 << 20, chunk_rows=1)
    m.load_graph(g.row_ptr, g.col, g.labels)
    star = m.query(3, [(0, 1), (0, 2)], [0, 0, 0])
    out = torch.empty(3 * d * (d - 1), dtype=torch.int32, device="cuda")
    for _ in range(2):
        with pytest.raises(gsm_lib.GsmError) as e:
            m.enumerate(star, out=out)
        out.fill_(-7)
        torch.cuda.synchronize()
        assert e.value.status == gsm_lib.GSM_ERR_BUDGET
        assert bool((out == -7).all())
    star.restrict(0, 0, 1)
    assert m.enumerate(star, out=out)[1] == d * (d - 1)
    assert out[:6].tolist() == [0, 2, 3, 0, 2, 4]
    m.close()


# widths that take 4-, 8- and 16-byte stores, matching orders that are canonical
# and others, last levels with and without checks
QUERIES = [(2, [(0, 1)]), (3, [(0, 1), (0, 2)]), (3, [(0, 1), (1, 2)]), (3, [(0, 1), (1, 2), (0, 2)]),
           (4, [(0, 1), (0, 2), (0, 3)]), (4, [(3, 2), (2, 1), (1, 0)]),
           (4, [(0, 1), (1, 2), (2, 3), (0, 3)]), (5, [(0, 1), (0, 2), (0, 3), (3, 4)]),
           (6, [(0, 1), (0, 2), (1, 2), (2, 3), (3, 4), (4, 5)])]
GUARD = 64  # ints that must not change on either side


@pytest.fixture(scope="module")
def listed(gsm_lib):
    n, rp, col = I.erdos_renyi(120, 420, seed=17)
    out = []
    for labels in (1, 2):
        g = I.make_graph(n, rp, col, np.arange(n, dtype=np.int32) % labels)
        items = []
        for k, edges in QUERIES:
            q = I.query_from_edges(k, edges, np.arange(k) % labels)
            count, rows, rc = oracle.match(g, q)
            assert rc == oracle.OK and count > 40
            items.append((q, rows))
        out.append((g, items))
    return out


def buffer(offset, cap, k):
    whole = torch.full((GUARD + offset + cap * k + GUARD,), -7, dtype=torch.int32, device="cuda")
    assert whole.data_ptr() % 16 == 0
    return whole, whole[GUARD + offset:]


def check(whole, offset, cap, rows, what):
    k = rows.shape[1]
    h = whole.cpu().numpy()
    a, n = GUARD + offset, min(cap, len(rows)) * k
    assert np.array_equal(h[a:a + n].reshape(-1, k), rows[:cap]), what
    assert (h[:a] == -7).all() and (h[a + cap * k:] == -7).all(), what


@pytest.mark.parametrize("opts", [{}, {"chunk_rows": 13}, {"chunk_rows": 50, "two_pass": True},
                                  {"mem_budget_bytes": 1 << 16}, {"hub_bitmap_bytes": -1,
                                                                  "chunk_rows": 1000}])
def test_device_buffers_of_any_alignment_and_room(gsm_lib, cuda, listed, opts):
    """Buffers on 4-byte boundaries, and buffers that end before, in the middle
    of and after the pieces a level is taken in: the rows are a prefix of the
    result, nothing beside them is written, and the whole result stays readable."""
    dev = gsm_lib.GSM_OUT_DEVICE
    for g, items in listed:
        m = gsm_lib.Matcher(device=0, **opts)
        m.load_graph(g.row_ptr, g.col, g.labels)
        for q, rows in items:
            Q, c = m.query(q.k, q.edges, q.labels), len(rows)
            for offset in range(4):
                for cap in (c + 3, c, c - 1, c // 2, c // 7, 1):
                    if offset and cap not in (c, c // 2):
                        continue
                    what = (opts, q.k, q.edges, offset, cap, c)
                    whole, out = buffer(offset, cap, q.k)
                    torch.cuda.synchronize()
                    count, st = gsm_lib.gsm_enumerate(m.ctx, Q.handle, out, cap, dev)
                    assert (count, st) == (c, gsm_lib.GSM_OK if cap >= c
                                           else gsm_lib.GSM_ERR_TRUNCATED), what
                    check(whole, offset, cap, rows, what)
                    kept = np.zeros((c, q.k), np.int32)
                    gsm_lib.gsm_last_rows(m.ctx, kept, 0, c, 0)
                    assert np.array_equal(kept, rows), what
        m.close()


@pytest.mark.parametrize("opts", [{}, {"host_workers": 1, "chunk_rows": 13},
                                  {"host_workers": 3, "copy_slots": 1, "chunk_rows": 40}])
def test_device_buffers_of_many(gsm_lib, cuda, listed, opts):
    for g, items in listed:
        m = gsm_lib.Matcher(device=0, **opts)
        m.load_graph(g.row_ptr, g.col, g.labels)
        jobs = [(q, rows, (j + t) % 4, (len(rows) + 3, len(rows), len(rows) // 2, len(rows) // 7)[t])
                for t in range(4) for j, (q, rows) in enumerate(items)]
        for part in (jobs, [j for j in jobs if j[3] >= len(j[1])]):
            bufs = [buffer(offset, cap, q.k) for q, _, offset, cap in part]
            Qs = [m.query(q.k, q.edges, q.labels) for q, *_ in part]
            torch.cuda.synchronize()
            counts, st = gsm_lib.gsm_enumerate_many(
                m.ctx, [Q.handle for Q in Qs], [out for _, out in bufs],
                [cap for *_, cap in part], gsm_lib.GSM_OUT_DEVICE)
            assert st == (gsm_lib.GSM_ERR_TRUNCATED if part is jobs else gsm_lib.GSM_OK)
            assert counts.tolist() == [len(rows) for _, rows, *_ in part]
            for (whole, _), (q, rows, offset, cap) in zip(bufs, part):
                check(whole, offset, cap, rows, (opts, q.k, q.edges, offset, cap, len(rows)))
            last = part[-1][1]
            kept = np.zeros_like(last)
            gsm_lib.gsm_last_rows(m.ctx, kept, 0, len(last), 0)
            assert np.array_equal(kept, last)
        m.close()
