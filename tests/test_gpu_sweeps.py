"""GPU: the grid-wide per-source kernel where its sweeps change form (backward sums pulled over a
level's own arcs or pushed over the next level's, path counts past 2^64 or not, bottom-up rows
around a lane's limit, bitmap words cut off), and the allocation-free entry's one-CTA teams."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1602_00963_gb300 as bc
from bcgpu import assert_bc_close, assert_sssp_equal, upload

pytestmark = pytest.mark.gpu

GRID = bc.BC_PATH_PLAIN | bc.BC_PLAIN_GRID


@pytest.fixture(scope="module")
def ctx():
    c = bc.bc_ctx_create(0)
    yield c
    bc.bc_destroy(c)


def layers(widths):
    """Consecutive layers of the given widths, completely joined."""
    off = np.concatenate([[0], np.cumsum(widths)])
    u, v = [], []
    for k in range(len(widths) - 1):
        i, j = np.meshgrid(np.arange(widths[k]), np.arange(widths[k + 1]), indexing="ij")
        u.append(off[k] + i.ravel())
        v.append(off[k + 1] + j.ravel())
    return gg.csr_from_edges(int(off[-1]), np.concatenate(u), np.concatenate(v), "layers-%d" % len(widths))


# shrinking tails push, growing ones pull; 2 and 16 wide for 70 and 20 layers pass 2^64 paths;
# 33 and 70 neighbours are rows beyond a lane's in a bottom-up level
SHAPES = [[1, 40, 60, 8, 2, 1], [1, 2, 8, 60, 40, 1], [1, 33, 1, 70, 1, 200, 3], [3] * 5 + [30, 30, 1, 1],
          [2] * 70, [1] + [16] * 20 + [4, 1, 1], [1, 1] + [16] * 20 + [64, 64, 2], [5, 500, 5, 500, 5], [32, 1, 31, 1]]


@pytest.mark.parametrize("si", range(len(SHAPES)))
def test_grid_kernel_layers(ctx, si):
    g = layers(SHAPES[si])
    h = upload(ctx, g)
    src = np.array([0, g.n - 1, g.n // 2, 0, 1], np.int32)
    want = oracle.bc(g, src)
    for flags in (GRID, GRID, GRID | bc.BC_NO_CD_REUSE):  # the second call starts at a later base
        got, st = bc.bc_sources(h, g.n, src, flags)
        assert_bc_close(got, want, what=f"{g.name} {flags}")
    for s in (0, g.n - 1):
        assert_sssp_equal(bc.bc_sssp(h, g.n, s, bc.BC_PLAIN_GRID), oracle.sssp(g, s), what=g.name)
    got, _ = bc.bc_sources(h, g.n, src, GRID)
    assert_bc_close(got, want, what=f"{g.name} after sssp")
    bc.bc_destroy(h)


def test_grid_kernel_leaves_and_isolated(ctx):
    """The 1-degree reduction on the grid-wide kernel: stars (a residual vertex with leaves and no
    edge), isolated vertices, and a leaf-rich graph."""
    stars = gg.csr_from_edges(40, [0, 0, 0, 5, 5, 9, 9, 9, 9], [1, 2, 3, 6, 7, 10, 11, 12, 13], "stars")
    for g in (stars, gg.attach_leaves(gg.rmat(8, 8, 4), 0.4, 5, 3)):
        h = upload(ctx, g)
        got, _ = bc.bc_exact(h, g.n, bc.BC_PRUNE_DEG1 | GRID)
        assert_bc_close(got, oracle.bc_exact(g), what=g.name)
        bc.bc_destroy(h)


@pytest.mark.parametrize("n,m,k", [(1, 0, 3), (31, 60, 1), (33, 60, 40), (1024, 8000, 120), (4096, 40000, 16),
                                   (4096, 40000, 1), (16384, 30000, 5), (30000, 200000, 2), (65536, 300000, 1)])
def test_noalloc_teams_and_grid(ctx, n, m, k):
    import torch
    g = gg.erdos_renyi(n, m, n + k) if m else gg.csr_from_edges(n, [], [])
    src = np.random.Generator(np.random.PCG64(k)).integers(0, n, k).astype(np.int32)
    want = oracle.bc(g, src)
    rp, ci = torch.from_numpy(g.row_ptr).cuda(), torch.from_numpy(g.col_idx).cuda()
    out = torch.full((n,), -7.0, dtype=torch.float64, device="cuda")
    bad = src.copy()
    bad[-1] = n
    with pytest.raises(bc.BCError) as e:  # refused on the device, the result left alone
        bc.bc_sources_noalloc(n, rp, ci, torch.from_numpy(bad).cuda(), out)
    assert e.value.status == bc.BC_EINVAL and bool((out == -7.0).all())
    for _ in range(2):
        bc.bc_sources_noalloc(n, rp, ci, torch.from_numpy(src).cuda(), out)
        assert_bc_close(out.cpu().numpy(), want, what=f"noalloc n={n} k={k}")
