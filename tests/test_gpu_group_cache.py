"""Multi-warp groups keep what they need of their eight cells when the grid holds
every active cell of a colour, and fetch it per phase when it does not.  Both
make the chain of the one-warp groups: two cells per axis (every cell in the
4 x 4 x 4 block twice), boxes whose blocks wrap, replicas of several sizes, and
grids on either side of the limit."""
import numpy as np
import pytest

from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _states(Ms, precision, schedules, sweeps, mix=W.PAPER_MIX):
    Ls = np.array([W.box_length(M) for M in Ms])
    st = [W.lattice_start(M, L, 40 + k, candidates=8, passes=1) for k, (M, L) in enumerate(zip(Ms, Ls))]
    one = len(Ms) == 1
    Ts = 1.5 if one else np.linspace(0.8, 2.5, len(Ms))
    seeds = 9 if one else np.arange(len(Ms), dtype=np.uint64) + np.uint64(9)
    out = []
    for W_, launch in schedules:
        h = F.Handle(float(Ls[0]) if one else Ls, np.concatenate([s[0] for s in st]), np.concatenate([s[1] for s in st]),
                     W.PAPER_POT, precision=precision, n_mol=None if one else np.array(Ms), warps_per_cell=W_,
                     launch_mode=launch)
        h.sweep(sweeps, Ts, mix, seeds)
        h.sync()
        stats = [{k: v for k, v in s.items() if k != "e_run"} for s in h.stats()]
        out.append((h.state_fixed(), stats))
        h.close()
    return out


def _same(out):
    for (state, stats) in out[1:]:
        assert all(np.array_equal(a, b) for a, b in zip(state, out[0][0]))
        assert stats == out[0][1]


@pytest.mark.parametrize("Ms", [[64], [300], [64, 300, 1000], [1000] * 8])
@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_cached_groups(Ms, precision):
    _same(_states(Ms, precision, [(1, 1), (2, 2), (4, 2), (8, 2)], 7, W.RIGID_MIX))


def test_grids_beyond_the_cells_they_hold():
    # 512 active cells: one per group with two warps, several with four and eight
    _same(_states([8000], "fp32", [(1, 2), (2, 2), (4, 2), (8, 2)], 4))
