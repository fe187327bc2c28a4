"""Memory budgets that are enough for the frontiers are enough for the call:
what only speeds a level up gives way, and no piece of a level takes the room
that a later level's smallest piece needs."""
import numpy as np
import pytest

import oracle
from paper_2003_01527_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def er(n, m, labels, seed):
    _, rp, col = I.erdos_renyi(n, m, seed=seed)
    lab = I.uniform_labels(n, labels, seed + 1) if labels > 1 else np.zeros(n, np.int32)
    return I.make_graph(n, rp, col, lab)


PATH4 = (4, [(0, 1), (1, 2), (2, 3)])
# graph, query, root range, bytes: about the frontiers of the largest row of each
# level beside the root candidates, with a third of them on top for scratch
CASES = {
    "hub": ("hub", 3, [(0, 1), (1, 2)], None, None, 142336),
    "hub_in_order": ("hub", 3, [(0, 1), (0, 2)], None, None, 142336),
    "path4": ("er1", *PATH4, None, (0, 150), 57088),
    "cycle4": ("er1", 4, [(0, 1), (1, 2), (2, 3), (0, 3)], None, None, 57088),
    "tailed_triangle": ("er1", 5, [(0, 1), (1, 2), (0, 2), (2, 3), (3, 4)], None, None, 84480),
    "star": ("er1", 5, [(0, 1), (0, 2), (0, 3), (0, 4)], None, (0, 3), 23552),
    "labelled_path4": ("er3", *PATH4, [0, 1, 2, 0], None, 31488),
    "labelled_star": ("er3", 4, [(0, 1), (1, 2), (1, 3)], [0, 1, 0, 1], None, 31488),
}


@pytest.fixture(scope="module")
def graphs():
    return {"hub": I.graph_from_edges(5001, [(0, v) for v in range(1, 5001)]),
            "er1": er(2000, 16000, 1, 5), "er3": er(3000, 30000, 3, 6)}


def open_query(gsm_lib, graphs, case, **opts):
    g, k, edges, labels, roots, _ = CASES[case]
    m = gsm_lib.Matcher(device=0, **opts)
    m.load_graph(graphs[g].row_ptr, graphs[g].col, graphs[g].labels)
    q = m.query(k, edges, labels)
    return m, q.restrict(0, *roots) if roots else q


@pytest.mark.parametrize("case", sorted(CASES))
def test_small_budgets(gsm_lib, cuda, graphs, case):
    g, k, edges, labels, roots, budget = CASES[case]
    want = oracle.match(graphs[g], I.query_from_edges(k, edges, labels), enumerate=False,
                        root_range=roots or (0, graphs[g].n))[0]
    m, q = open_query(gsm_lib, graphs, case)
    rows, count = m.enumerate(q)
    assert count == want
    m.close()
    for opts in ({}, {"hub_bitmap_bytes": -1}):
        m, q = open_query(gsm_lib, graphs, case, mem_budget_bytes=budget, **opts)
        assert m.count(q) == want
        got, count = m.enumerate(q)
        assert count == want and np.array_equal(got, rows)
        assert m.last_run_stats()["peak_bytes"] <= budget
        m.close()


@pytest.mark.parametrize("case", ["cycle4", "tailed_triangle"])
def test_every_larger_budget_is_enough_too(gsm_lib, cuda, graphs, case):
    m, q = open_query(gsm_lib, graphs, case)
    want = m.count(q)
    m.close()
    least = CASES[case][-1]
    for budget in range(least, 3 * least, 1536):
        m, q = open_query(gsm_lib, graphs, case, mem_budget_bytes=budget)
        assert m.count(q) == want, budget
        assert m.enumerate(q, cap_rows=0)[1] == want, budget
        m.close()


def test_too_small_a_budget_is_still_refused(gsm_lib, cuda, graphs):
    for case in ("hub", "tailed_triangle"):
        m, q = open_query(gsm_lib, graphs, case, mem_budget_bytes=16384)
        with pytest.raises(gsm_lib.GsmError) as e:
            m.enumerate(q, cap_rows=0)
        assert e.value.status == gsm_lib.GSM_ERR_BUDGET
        m.close()
