"""GPU: the per-CTA kernel's workspace over calls in a row: more sources each time, and calls of
different layouts taking turns, neither of which may allocate it anew each time."""
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


def free_bytes():
    import torch
    return torch.cuda.mem_get_info()[0]


def changes(values):
    return int(np.count_nonzero(np.diff(values)))


def test_growing_number_of_sources(ctx):
    """33 to 150 sources on state in global memory, 1.9 MB per CTA: growth by doubling changes the
    free memory three times (33, 66, 132, 152 or more); the exact fit at nearly every call."""
    g = gg.erdos_renyi(60000, 90000, 7)
    h = upload(ctx, g)
    src = np.arange(150, dtype=np.int32) * 397
    free = []
    for k in range(33, 151):
        got, _ = bc.bc_sources(h, g.n, src[:k], CTA)
        free.append(free_bytes())
    assert changes(free) <= 3
    assert_bc_close(got, oracle.bc(g, src, nthreads=8), what="last call")
    few, _ = bc.bc_sources(h, g.n, src[:3], CTA)  # on a workspace of many CTAs
    assert_bc_close(few, oracle.bc(g, src[:3]), what="few sources")
    bc.bc_destroy(h)


def test_layouts_taking_turns(ctx):
    """Runs of 2-degree triples (two states in global memory) and of single sources (state in shared
    memory, more CTAs) on one graph."""
    g = gg.subdivide_edges(gg.ba_pref_attach(1500, 3), 0.1, 5)
    h = upload(ctx, g)
    want = oracle.bc_exact(g, nthreads=8)
    free, first = [], None
    for turn in range(4):
        a, _ = bc.bc_exact(h, g.n, bc.BC_DEG2)
        free.append(free_bytes())
        b, _ = bc.bc_exact(h, g.n, CTA)
        free.append(free_bytes())
        first = first or (a, b)
        assert np.array_equal(a, first[0]) and np.array_equal(b, first[1])
    assert_bc_close(a, want, what="triples")
    assert_bc_close(b, want, what="single sources")
    assert changes(free[1:]) == 0  # after one call of each the workspace serves both
    bc.bc_destroy(h)


def test_row_records_after_a_shared_layout(ctx):
    """A call with its state in global memory builds its row records (one launch more) whatever
    workspace an earlier call of another layout left."""
    g = gg.subdivide_edges(gg.ba_pref_attach(1500, 3), 0.1, 5)
    launches = []
    for before in (None, CTA):
        h = upload(ctx, g)
        if before is not None:
            bc.bc_exact(h, g.n, before)
        launches.append(bc.bc_exact(h, g.n, bc.BC_DEG2)[1]["kernel_launches"])
        bc.bc_destroy(h)
    assert launches == [launches[0]] * 2 and launches[0] >= 3
