"""GPU: the per-source kernel that runs one source per CTA, at the edges of its dispatch: state in
shared memory with and without its queue, in global memory, narrow graphs; rows around the
degrees at which a lane, eight lanes or a warp take a vertex, with and without path counts past
2^64 in each; levels longer than the shared-memory ring; calls in a row on one workspace."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1602_00963_gb300 as bc
from bcgpu import assert_bc_close, assert_sssp_equal, upload

pytestmark = pytest.mark.gpu

CTA = bc.BC_PATH_PLAIN | bc.BC_PLAIN_CTA


@pytest.fixture(scope="module")
def ctx():
    c = bc.bc_ctx_create(0)
    yield c
    bc.bc_destroy(c)


def layered(width, layers, n=0):
    """Consecutive layers of `width` vertices, completely joined: inner degrees 2 * width, width^l
    paths to layer l.  Padded with isolated vertices to n."""
    i, j = np.meshgrid(np.arange(width), np.arange(width), indexing="ij")
    off = np.arange(layers - 1)[:, None] * width
    u = (off + i.ravel()).ravel()
    v = (off + width + j.ravel()).ravel()
    return gg.csr_from_edges(max(n, width * layers), u, v, f"layered-{width}x{layers}")


# widths: degrees 2, 4, 6, 8, 10, 16, 18, 32, 34, 64, 66, 130; as many layers as pass 2^64 paths
@pytest.mark.parametrize("n", [0, 30000], ids=["shared", "global"])
@pytest.mark.parametrize("width", [1, 2, 3, 4, 5, 8, 9, 16, 17, 32, 33, 65])
def test_rows_and_overflow_at_each_degree(ctx, width, n):
    layers = 80 if width <= 2 else int(64 / np.log2(width)) + 4
    for k in (5, layers):  # without and (width > 1) with path counts past 2^64
        g = layered(width, k, n)
        h = upload(ctx, g)
        src = np.array([0, width * k - 1, width * (k // 2), 0], np.int32)
        for _ in range(2):  # a second call on the same workspace
            got, st = bc.bc_sources(h, g.n, src, CTA)
            assert_bc_close(got, oracle.bc(g, src), what=f"{g.name} n={g.n}")
            assert (st["sigma_overflow_sources"] > 0) == (width > 1 and k == layers)
            assert st["max_depth"] == k - 1
        assert_sssp_equal(bc.bc_sssp(h, g.n, 0), oracle.sssp(g, 0), what=g.name)
        bc.bc_destroy(h)


# the sizes at which the queue, then the state leave shared memory, and their neighbours; ids and
# levels at the end of their 16 bits are covered by the path graphs
@pytest.mark.parametrize("n", [33, 4099, 18915, 18916, 18917, 22653, 22654, 22655, 40001])
def test_sizes(ctx, n):
    for g in (gg.erdos_renyi(n, min(3 * n, n * (n - 1) // 4), n), gg.ba_pref_attach(n, n) if n < 25000 else gg.path_graph(n)):
        h = upload(ctx, g)
        src = np.unique(np.array([0, 1, n // 2, n - 1], np.int32))
        got, _ = bc.bc_sources(h, g.n, src, CTA)
        assert_bc_close(got, oracle.bc(g, src), what=g.name)
        s = int(src[-1])
        assert_sssp_equal(bc.bc_sssp(h, g.n, s, bc.BC_PLAIN_CTA), oracle.sssp(g, s), what=g.name)
        bc.bc_destroy(h)


def test_deepest_levels_in_shared_memory(ctx):
    """A path of 22,625 vertices (levels close to the limit of n) with a hub of 30 arcs at its
    start, so that the graph is not narrow."""
    n = 22654
    g = gg.csr_from_edges(n, np.concatenate([np.arange(n - 30), np.zeros(29, np.int64)]),
                          np.concatenate([np.arange(1, n - 29), np.arange(n - 29, n)]), "path-hub")
    h = upload(ctx, g)
    src = np.array([0, n - 30, n - 1], np.int32)
    got, st = bc.bc_sources(h, g.n, src, CTA)
    assert st["max_depth"] == n - 29
    assert_bc_close(got, oracle.bc(g, src), what=g.name)
    assert_sssp_equal(bc.bc_sssp(h, g.n, n - 1), oracle.sssp(g, n - 1), what=g.name)
    bc.bc_destroy(h)


def test_levels_beyond_the_ring(ctx):
    """A hub with more than 2048 neighbours (the ring), state in global memory, each neighbour
    with a private and a shared second neighbour."""
    m = 9001
    hub = np.zeros(m, np.int64)
    mid = np.arange(1, m + 1)
    g = gg.csr_from_edges(3 * m + 2, np.concatenate([hub, mid, mid]),
                          np.concatenate([mid, mid + m, np.full(m, 2 * m + 1)]), "wide")
    h = upload(ctx, g)
    src = np.array([0, 5, 2 * m + 1, m + 7], np.int32)
    got, _ = bc.bc_sources(h, g.n, src, CTA)
    assert_bc_close(got, oracle.bc(g, src), what=g.name)
    bc.bc_destroy(h)


def test_deg2_with_overflow_and_without(ctx):
    """2-degree triples whose DAGs pass 2^64 paths on one or both sides, and a chain-rich road."""
    wide = layered(4, 40)
    u, v = wide.edges()
    n = wide.n  # degree-2 vertices: one across the two ends, one beside the middle
    g = gg.csr_from_edges(n + 2, np.concatenate([u, [n, n, n + 1, n + 1]]),
                          np.concatenate([v, [0, n - 1, n // 2, n // 2 + 4]]), "layered-deg2")
    road = gg.attach_leaves(gg.subdivide_edges(gg.grid2d(18, 15, 4, 0.1), 0.4, 5), 0.15, 6, 2)
    for x in (g, road):
        h = upload(ctx, x)
        want = oracle.bc_exact(x)
        for flags in (bc.BC_DEG2, bc.BC_DEG2 | bc.BC_PRUNE_DEG1, 0):
            got, _ = bc.bc_exact(h, x.n, flags)
            assert_bc_close(got, want, what=f"{x.name} {flags}")
        bc.bc_destroy(h)


def test_tight_budget_without_row_records(ctx):
    """A context budget that leaves room for the graph and one CTA's state alone."""
    g = gg.grid2d(220, 140, 3, 0.1)
    budget = (g.n + 1) * 4 + g.nnz * 4 + g.n * 8 * 2 + 16 + g.n * 34
    c = bc.bc_ctx_create(0, budget)
    h = upload(c, g)
    src = np.array([3, 1000, g.n - 1], np.int32)
    got, _ = bc.bc_sources(h, g.n, src, CTA)
    assert_bc_close(got, oracle.bc(g, src), what="tight budget")
    bc.bc_destroy(h)
    bc.bc_destroy(c)
