"""GPU: the scratch that picks the source order's landmarks counts against the context's HBM budget: where
the budget has no room for it, it is what is refused."""
import re

import numpy as np
import pytest

import graphgen as gg
import paper_1602_00963_gb300 as bc
from bcgpu import upload

pytestmark = pytest.mark.gpu


def test_landmark_scratch_is_in_the_budget():
    import torch
    n = 1 << 18
    g = gg.erdos_renyi(n, 2 * n, 1)
    src = torch.arange(4 * 32, dtype=torch.int32, device="cuda")  # four tiles: ordered by locality
    out = torch.zeros(n, dtype=torch.float64, device="cuda")
    first_refused = []
    for budget in range(0, 40 * n, 2 * n):  # the graph takes 20 n, the scratch 8 n, the distances 160 n
        c = bc.bc_ctx_create(0, max(budget, 1))
        try:
            h = upload(c, g)
            with pytest.raises(bc.BCError) as e:
                bc.bc_sources(h, n, src, bc.BC_PATH_TILED | bc.BC_TILE(32), out)
            assert e.value.status == bc.BC_ENOMEM
            first_refused.append(int(re.search(r"allocation of (\d+) bytes", str(e.value)).group(1)))
        except bc.BCError as e:  # no room for the graph
            assert e.status == bc.BC_ENOMEM
        bc.bc_destroy(c)
    assert any(8 * n <= b < 9 * n for b in first_refused), first_refused
