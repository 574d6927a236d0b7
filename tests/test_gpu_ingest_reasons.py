"""GPU: a refused graph's message names the invariant that it breaks (where rows break several, the one
listed last: ends, order of the offsets, range, self-loop, order in a row, symmetry)."""
import numpy as np
import pytest

import paper_1602_00963_gb300 as bc

pytestmark = pytest.mark.gpu

ENDS, OFFSETS, RANGE, LOOP, ORDER, ONE_WAY = (
    "row_ptr[0] != 0 or row_ptr[n] != nnz", "row_ptr decreases", "column index out of range", "self-loop",
    "row not strictly increasing (duplicate edge or unsorted)", "CSR is not symmetric")


@pytest.mark.parametrize("rp,ci,why", [
    ([1, 1], [], ENDS), ([0, 0, 2], [], ENDS), ([0, 2, 0], [0, 1], LOOP), ([0, 1, 0, 0], [], OFFSETS),
    ([0, 2], [3, 4], RANGE), ([0, 2], [-1, 0], RANGE), ([0, 2], [0, 0], LOOP), ([0, 2, 4], [1, 1, 0, 0], ORDER),
    ([0, 2, 3, 4], [2, 1, 0, 0], ONE_WAY), ([0, 1, 2, 2], [1, 2], ONE_WAY), ([0, 1, 2, 4], [2, 2, 0, 1], None)])
def test_reason(rp, ci, why):
    c = bc.bc_ctx_create(0)
    rp, ci = np.array(rp, np.int32), np.array(ci, np.int32)
    if why is None:
        bc.bc_destroy(bc.bc_graph_create(c, rp.size - 1, rp, ci, ci.size, bc.BC_VALIDATE))
    else:
        with pytest.raises(bc.BCError) as e:
            bc.bc_graph_create(c, rp.size - 1, rp, ci, ci.size, bc.BC_VALIDATE)
        assert e.value.status == bc.BC_EINVAL
        assert str(e.value) == f"BC_EINVAL: bc_graph_create: invalid CSR: {why}"
    bc.bc_destroy(c)
