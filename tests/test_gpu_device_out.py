"""Listings into device memory: what is written there, and until when."""
import numpy as np
import pytest
import torch

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
