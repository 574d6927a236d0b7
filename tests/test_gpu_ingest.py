"""GPU: graph ingest (BC_VALIDATE) and the 1-degree reduction at the sizes where their arc-parallel
kernels can go wrong: chunks of 1024 arcs, words of 32, rows longer than both, long runs of empty
rows, hubs, no arcs at all."""
import numpy as np
import pytest

import graphgen as gg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_1602_00963_gb300 as bc
    c = bc.bc_ctx_create(0)
    yield c
    bc.bc_destroy(c)


def scattered(n, m, gap, seed):
    """gnm on every gap-th vertex: runs of empty rows between the others, also first and last."""
    g = gg.erdos_renyi(n, m, seed)
    u, v = g.edges()
    return gg.csr_from_edges(n * gap + gap, u * gap + gap // 2, v * gap + gap // 2, f"scattered-{gap}")


GRAPHS = [
    lambda: gg.csr_from_edges(1, [], []),
    lambda: gg.csr_from_edges(70, [], []),
    lambda: gg.path_graph(2),
    lambda: gg.path_graph(513),
    lambda: gg.path_graph(514),
    lambda: gg.star_graph(3000),
    lambda: gg.complete_graph(33),
    lambda: gg.complete_graph(90),
    lambda: gg.random_tree(2000, 3),
    lambda: scattered(300, 1500, 77, 1),
    lambda: scattered(40, 60, 4001, 2),
    lambda: gg.rmat(12, 16, 9),
    lambda: gg.attach_leaves(gg.rmat(10, 8, 4), 0.3, 5, 40),
]


@pytest.mark.parametrize("make", GRAPHS)
def test_valid_graphs_are_accepted_and_pruned(ctx, make):
    import paper_1602_00963_gb300 as bc
    g = make()
    h = bc.bc_graph_create(ctx, g.n, g.row_ptr, g.col_idx, g.nnz, bc.BC_VALIDATE)
    omega, removed, rrp, rci = bc.bc_prune(h, g.n, g.nnz)
    bc.bc_destroy(h)
    deg = g.degrees()
    row = np.repeat(np.arange(g.n), deg)
    first = np.where(deg == 1, g.col_idx[np.minimum(g.row_ptr[:-1], max(g.nnz - 1, 0))] if g.nnz else 0, 0)
    rem = (deg == 1) & (deg[first] >= 2)
    keep = ~rem[row] & ~rem[g.col_idx]
    np.testing.assert_array_equal(removed.astype(bool), rem)
    np.testing.assert_array_equal(omega, np.bincount(first[rem], minlength=g.n))
    np.testing.assert_array_equal(rci, g.col_idx[keep])
    np.testing.assert_array_equal(rrp, np.concatenate([[0], np.cumsum(np.bincount(row[keep], minlength=g.n))]))


def broken(kind):
    """A graph of 3000 vertices with one invariant broken somewhere in the middle."""
    g = gg.rmat(12, 8, 6)
    rp, ci = g.row_ptr.copy(), g.col_idx.copy()
    u = int(np.argmax(g.degrees()))
    a, b = int(rp[u]), int(rp[u + 1])
    e = a + (b - a) // 2
    if kind == "range":
        ci[b - 1] = g.n
    elif kind == "negative":
        ci[a] = -1
    elif kind == "self-loop":
        ci[np.searchsorted(ci[a:b], u) + a - 1] = u  # between a smaller and a larger neighbour
    elif kind == "duplicate":
        ci[e] = ci[e - 1]
    elif kind == "unsorted":
        ci[e], ci[e - 1] = ci[e - 1], ci[e]
    elif kind == "decreasing":
        rp[u] = rp[u + 1] + 1
    elif kind == "end":
        rp[-1] -= 2
    else:  # one arc's reverse replaced by an arc to another vertex, rows still sorted
        w = int(ci[e])
        pos = int(rp[w] + np.searchsorted(ci[rp[w]:rp[w + 1]], u))
        lo = int(ci[pos - 1]) if pos > rp[w] else -1
        hi = int(ci[pos + 1]) if pos + 1 < rp[w + 1] else g.n
        free = [x for x in range(lo + 1, hi) if x not in (u, w)]
        assert free
        ci[pos] = free[0]
    return g.n, rp, ci


@pytest.mark.parametrize("kind,text", [
    ("range", "out of range"), ("negative", "out of range"), ("self-loop", "invalid CSR"),
    ("duplicate", "invalid CSR"), ("unsorted", "invalid CSR"), ("decreasing", "invalid CSR"),
    ("end", "invalid CSR"), ("one-way", "not symmetric")])
def test_broken_graphs_are_refused(ctx, kind, text):
    import paper_1602_00963_gb300 as bc
    n, rp, ci = broken(kind)
    with pytest.raises(bc.BCError) as e:
        bc.bc_graph_create(ctx, n, rp, ci, ci.size, bc.BC_VALIDATE)
    assert e.value.status == bc.BC_EINVAL
    assert "invalid CSR" in str(e.value) and (text in str(e.value) or "symmetric" in str(e.value))
