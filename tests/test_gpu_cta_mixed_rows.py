"""GPU: the per-CTA kernel with its state in global memory, where rows of at most four arcs (a lane
adds their extended-range sums from registers) share a warp with longer ones (the warp's arc loop
then goes on after the short rows are done), with path counts past 2^64."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1602_00963_gb300 as bc
from bcgpu import assert_bc_close, upload

pytestmark = pytest.mark.gpu

CTA = bc.BC_PATH_PLAIN | bc.BC_PLAIN_CTA


@pytest.fixture(scope="module")
def ctx():
    c = bc.bc_ctx_create(0)
    yield c
    bc.bc_destroy(c)


def mixed(w, h, seed, diagonals=0.0, leaves=0.0, max_leaves=4, bridges=0.0, n=0):
    """A w x h grid; a fraction of its cells get a diagonal, another a vertex of degree 2 across the
    other diagonal (as long as the two grid paths beside it), a fraction of the vertices leaves.
    Padded with isolated vertices to n."""
    rng = np.random.Generator(np.random.PCG64(seed))
    g = gg.grid2d(w, h)
    u, v = g.edges()
    x, y = np.meshgrid(np.arange(w - 1), np.arange(h - 1), indexing="ij")
    cell = (y * w + x).ravel()
    d = cell[rng.random(cell.size) < diagonals]
    b = cell[rng.random(cell.size) < bridges]
    c = w * h + np.arange(b.size)
    u = np.concatenate([u, d, b + 1, b + w])
    v = np.concatenate([v, d + w + 1, c, c])
    hub = np.flatnonzero(rng.random(w * h) < leaves)
    hub = np.repeat(hub, rng.integers(1, max_leaves + 1, hub.size))
    leaf = w * h + b.size + np.arange(hub.size)
    total = w * h + b.size + hub.size
    return gg.csr_from_edges(max(total, n), np.concatenate([u, hub]), np.concatenate([v, leaf]), f"mixed-{w}x{h}")


# largest degree 8 (narrow kernel) and up to 16 (a lane takes rows of up to 16 arcs); every graph
# has n above what the state in shared memory is used for
@pytest.mark.parametrize("make", [
    lambda: mixed(90, 90, 1, diagonals=0.05),
    lambda: mixed(90, 90, 2, leaves=0.1),
    lambda: mixed(84, 84, 3, diagonals=0.03, leaves=0.05, max_leaves=2, bridges=0.05),
    lambda: mixed(90, 90, 4, leaves=0.1, max_leaves=12, n=30000),
    lambda: mixed(90, 90, 5, diagonals=0.05, leaves=0.1, max_leaves=8, n=30000),
], ids=["diagonals-narrow", "leaves-narrow", "all-narrow", "leaves-16", "all-16"])
def test_short_and_long_rows_in_one_warp(ctx, make):
    g = make()
    src = np.array([0, 1, 89, 83, 45, 90 * 40 + 3], np.int32)  # 89, 83: corners that no diagonal brings nearer
    h = upload(ctx, g)
    got, st = bc.bc_sources(h, g.n, src, CTA)
    bc.bc_destroy(h)
    assert st["sigma_overflow_sources"] > 0
    assert_bc_close(got, oracle.bc(g, src), what=g.name)


@pytest.mark.parametrize("make", [
    lambda: mixed(44, 44, 6, diagonals=0.02, bridges=0.05),
    lambda: mixed(44, 44, 7, leaves=0.1, max_leaves=10, bridges=0.08),
], ids=["narrow", "16"])
def test_two_degree_runs(ctx, make):
    g = make()
    want = oracle.bc_exact(g, nthreads=8)
    h = upload(ctx, g)
    for flags in (bc.BC_DEG2, bc.BC_DEG2 | bc.BC_PRUNE_DEG1):
        got, st = bc.bc_exact(h, g.n, flags)
        assert st["sigma_overflow_sources"] > 0
        assert_bc_close(got, want, what=f"{g.name} {flags}")
    bc.bc_destroy(h)
