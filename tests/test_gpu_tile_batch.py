"""GPU: tiles launched in a row without waiting: more tiles than a batch holds, and batches in which
a tile in the middle has to run again (path counts past 2^64, an active list that overflows)."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1602_00963_gb300 as bc
from bcgpu import assert_bc_close, upload

pytestmark = pytest.mark.gpu

T32 = bc.BC_PATH_TILED | bc.BC_TILE(32)


@pytest.fixture(scope="module")
def ctx():
    c = bc.bc_ctx_create(0)
    yield c
    bc.bc_destroy(c)


def union(a, b):
    u, v = a.edges()
    x, y = b.edges()
    return gg.csr_from_edges(a.n + b.n, np.concatenate([u, x + a.n]), np.concatenate([v, y + a.n]), "union")


def test_more_tiles_than_a_batch(ctx):
    g = gg.rmat(11, 8, 5)
    src = np.random.Generator(np.random.PCG64(1)).integers(0, g.n, 32 * 66 + 7).astype(np.int32)
    want = oracle.bc(g, src, nthreads=8)
    h = upload(ctx, g)
    for flags in (T32 | bc.BC_KEEP_ORDER, T32):
        got, st = bc.bc_sources(h, g.n, src, flags)
        assert st["sources"] == src.size
        assert_bc_close(got, want, what=f"batch {flags}")
    again, _ = bc.bc_sources(h, g.n, src, T32)
    assert np.array_equal(got, again)
    bc.bc_destroy(h)


def test_overflow_in_the_middle_of_a_batch(ctx):
    """Tiles 0, 1 and 3 in a component of few paths, tile 2 in a grid whose counts pass 2^64."""
    a, b = gg.rmat(9, 8, 2), gg.grid2d(40, 40)
    g = union(a, b)
    rng = np.random.Generator(np.random.PCG64(3))
    small = np.flatnonzero(a.degrees() > 0)
    src = np.concatenate([rng.choice(small, 64), a.n + rng.integers(0, b.n, 32), rng.choice(small, 40)]).astype(np.int32)
    want = oracle.bc(g, src)
    h = upload(ctx, g)
    for _ in range(2):  # the second call starts in the extended range
        got, st = bc.bc_sources(h, g.n, src, T32 | bc.BC_KEEP_ORDER)
        assert_bc_close(got, want, what="middle overflow")
        assert 0 < st["sigma_overflow_sources"] <= 32 and st["sources"] == src.size
    bc.bc_destroy(h)


def test_active_list_grows_in_the_middle_of_a_batch(ctx):
    """A path: the tile whose 32 sources lie far apart has every vertex in the active list at up
    to 32 levels, past the list's first capacity of 4 n + 1024 entries; the tiles around it fit."""
    g = gg.path_graph(4001)
    src = np.concatenate([np.full(32, 7), np.arange(32) * 125, np.full(32, 4000), [0, 1]]).astype(np.int32)
    want = oracle.bc(g, src)
    h = upload(ctx, g)
    got, st = bc.bc_sources(h, g.n, src, T32 | bc.BC_KEEP_ORDER)
    assert st["sources"] == src.size and st["max_depth"] == 4000
    assert_bc_close(got, want, what="list growth")
    bc.bc_destroy(h)
