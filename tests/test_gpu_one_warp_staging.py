"""One-warp groups of a persistent launch stage their neighbourhood by bulk
copies, which read records that other blocks wrote in the same launch (commits
of neighbour cells, the order pass).  Those reads have to see the writes: over
many sweeps the chain is that of kernels which meet at kernel boundaries, and of
the groups that stage by ordinary loads."""
import numpy as np
import pytest

from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# 64 and 1000 molecules: every cell waits for neighbours that have only just
# committed; 20000: several cells per warp, the sizes one-warp groups are for
@pytest.mark.parametrize("M,precision,sweeps", [(64, "fp32", 300), (1000, "fp32", 150), (1000, "fp64", 20), (20000, "fp32", 60)])
def test_bulk_copies_see_the_records_of_the_same_launch(M, precision, sweeps):
    L = W.box_length(M)
    xyz, t = W.lattice_start(M, L, 5, candidates=8, passes=1)
    states = []
    for wpc, launch in ((1, 2), (1, 1), (2, 2)):
        h = F.Handle(L, xyz, t, W.PAPER_POT, precision=precision, warps_per_cell=wpc, launch_mode=launch)
        h.sweep(sweeps, 1.5, W.PAPER_MIX, 17)
        h.sync()
        states.append(h.state_fixed())
        h.close()
    for s in states[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(s, states[0]))
