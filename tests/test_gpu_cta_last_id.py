"""GPU: the per-CTA kernel at its largest n, 2^24, where a vertex id fills the 24 bits that a queue entry
has for it, and all eight successor bits above them are set too."""
import numpy as np
import pytest

import graphgen as gg
import oracle
import paper_1602_00963_gb300 as bc
from bcgpu import assert_bc_close, upload

pytestmark = pytest.mark.gpu

CTA = bc.BC_PATH_PLAIN | bc.BC_PLAIN_CTA


# side: leaves of the last vertex's parent, so that the last vertex lies in a level's first window
# of entries or in a later one
@pytest.mark.parametrize("side", [0, 700])
def test_last_vertex_with_eight_successors(side):
    n = 1 << 24
    last, s, t = n - 1, n - 2, n - 3
    k = np.arange(8)
    # last: eight neighbours one level deeper (each with a leaf of its own), its parent s the ninth
    u = np.concatenate([np.full(8, last), [last, s], k, np.full(side, s)])
    v = np.concatenate([k, [s, t], 100 + k, 1000 + np.arange(side)])
    g = gg.csr_from_edges(n, u, v, f"last-{side}")
    src = np.array([s, t, 100, 0, last], np.int32)  # the last vertex on levels 1, 2, 2, 1 and 0
    c = bc.bc_ctx_create(0, 3 << 30)
    h = upload(c, g)
    got, st = bc.bc_sources(h, n, src, CTA)
    bc.bc_destroy(h)
    bc.bc_destroy(c)
    assert st["max_depth"] == 4 and st["sources"] == src.size
    assert_bc_close(got, oracle.bc(g, src), what=g.name)
