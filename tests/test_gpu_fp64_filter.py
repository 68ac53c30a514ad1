"""FP64 mode refuses attempts by a rigorous FP32 bound where it can.  A logged
sweep takes the FP64 sum for every attempt, so a handle that logs and one that
does not must agree in everything: state, running energy bit for bit, and
every counter (pair_interactions among them)."""
import numpy as np
import pytest

from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SOFT = (0.9, 1.0, 1.1, 1e-25, 33.75, 1.5)     # eps far below FP32's normal range for products: no FP32 refusals
ODD = (0.5, 1.0, 1.4, 3.0, 5.0, 1.9)          # another potential inside it


def _pair(M, pot, W_, launch, n_cells=0, gap=0.0):
    L = W.box_length(M)
    xyz, t = W.lattice_start(M, L, M)
    return [F.Handle(L, xyz, t, pot, precision="fp64", warps_per_cell=W_, launch_mode=launch, n_cells=n_cells,
                     recheck_gap=gap) for _ in range(2)]


def _same(a, b, T, mix, n, seed):
    a.sweep(n, T, mix, seed)
    b.sweep_logged(n, T, mix, seed)
    for x, y in zip(a.state_fixed(), b.state_fixed()):
        assert np.array_equal(x, y)
    sa, sb = a.stats()[0], b.stats()[0]
    assert sa == sb
    assert sa["fp64_rechecks"] == 0
    a.close()
    b.close()


@pytest.mark.parametrize("mix", [W.PAPER_MIX, W.LOCAL_MIX, W.RIGID_MIX])
@pytest.mark.parametrize("W_,launch", [(1, 1), (1, 2), (2, 2), (4, 2), (8, 2), (4, 1)])
def test_filtered_chain_is_the_chain_of_all_sums(mix, W_, launch):
    _same(*_pair(300, W.PAPER_POT, W_, launch), 0.9, mix, 12, 5)


@pytest.mark.parametrize("M,T", [(64, 3.0), (64, 0.02), (1000, 0.75)])
def test_filtered_chain_over_sizes_and_temperatures(M, T):
    _same(*_pair(M, W.PAPER_POT, 0, 0), T, W.RIGID_MIX, 10, 7)


@pytest.mark.parametrize("pot,T", [(SOFT, 1e-25), (ODD, 2.0), (W.PAPER_POT, 1e-24)])
def test_parameters_at_and_beyond_the_range_of_the_bound(pot, T):
    _same(*_pair(216, pot, 0, 0, n_cells=2), T, W.RIGID_MIX, 6, 9)


def test_recheck_gap_does_not_loosen_the_fp64_chain():
    _same(*_pair(216, W.PAPER_POT, 0, 0, gap=1e-12), 1.0, W.PAPER_MIX, 10, 3)
