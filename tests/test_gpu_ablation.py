"""GPU: the prefix-reuse ablation changes the reuse alone.  The backward sweep takes each level by the
same rule (pulled over its own arcs, or pushed over the next level's) and scans again the prefix that
it is about to read, each level's once."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

RUN = """
import sys
import numpy as np
import paper_1602_00963_gb300 as bc
from test_gpu_sweeps import layers
g = layers([int(x) for x in sys.argv[1].split(",")])
c = bc.bc_ctx_create(0)
h = bc.bc_graph_create(c, g.n, g.row_ptr, g.col_idx, g.nnz, bc.BC_VALIDATE)
bc.bc_sources(h, g.n, np.array([0], np.int32), bc.BC_PATH_PLAIN | bc.BC_PLAIN_GRID | int(sys.argv[2]))
"""
RESCAN_PHASE = 8


# arcs of levels 0, 1, ...: 40, 2440, 2880, 496, 18, 2: level 1 is pulled, the others pushed to;
# 2, 18, 496, 2880, 2440, 40: only level 4 is pushed to; 100, 6100, 6120, 240, 240, 120: levels 4 and 2
# are pushed to, level 2 from level 3, whose prefix was scanned when it was pulled
@pytest.mark.parametrize("widths,scanned", [("1,40,60,8,2,1", [5, 4, 3, 1]), ("1,2,8,60,40,1", [5, 3, 2, 1]),
                                            ("1,100,60,2,60,2", [5, 3, 1])])
def test_scans_the_prefix_each_step_reads(tmp_path, widths, scanned):
    import paper_1602_00963_gb300 as bc
    here = os.path.dirname(os.path.abspath(__file__))
    for flag, want in ((0, []), (bc.BC_NO_CD_REUSE, scanned)):
        out = tmp_path / f"trace{flag}"
        env = dict(os.environ, BC_TRACE_FILE=str(out),
                   PYTHONPATH=os.pathsep.join([os.path.dirname(here), here, os.environ.get("PYTHONPATH", "")]))
        subprocess.run([sys.executable, "-c", RUN, widths, str(flag)], env=env, check=True, timeout=300)
        rows = [line.split(",") for line in out.read_text().split()]
        assert [int(r[1]) for r in rows if int(r[0]) == RESCAN_PHASE] == want
