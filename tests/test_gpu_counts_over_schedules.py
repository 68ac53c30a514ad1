"""Every counter is that of the serial order of the attempts, whatever the warps
per cell: also pair_interactions, which takes in the refused attempts.  Small
dense replicas far from equilibrium, two cells per axis, many attempts of one
cell close together: an attempt that breaks a bond may lie near an earlier one
of its round that was accepted."""
import numpy as np
import pytest

from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _start(Ms, seed):
    Ls = np.array([W.box_length(int(M)) for M in Ms])
    st = [W.lattice_start(int(M), L, seed + k, candidates=4, passes=1) for k, (M, L) in enumerate(zip(Ms, Ls))]
    return Ls, np.concatenate([s[0] for s in st]), np.concatenate([s[1] for s in st])


@pytest.mark.parametrize("precision,sweeps", [("fp32", 200), ("fp64", 30)])
def test_counters_do_not_depend_on_the_warps_per_cell(precision, sweeps):
    Ms = np.random.default_rng(1).integers(66, 120, 146).astype(np.int32)
    Ts = np.random.default_rng(2).uniform(0.75, 3.0, 146)
    Ls, xyz, t = _start(Ms, 40)
    seeds = np.arange(146, dtype=np.uint64) + np.uint64(9)
    ref = None
    for wpc in (1, 2, 4, 8):
        h = F.Handle(Ls, xyz, t, W.PAPER_POT, precision=precision, n_mol=Ms, warps_per_cell=wpc)
        h.sweep(sweeps, Ts, W.PAPER_MIX, seeds)
        h.sync()
        # (the running energy adds the same terms in another order)
        got = [{k: v for k, v in s.items() if k != "e_run"} for s in h.stats()]
        h.close()
        ref = ref or got
        assert got == ref, wpc


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_counters_do_not_depend_on_the_autotuner(precision):
    Ls, xyz, t = _start([90], 30)
    got = []
    for tune in (False, True):
        h = F.Handle(float(Ls[0]), xyz, t, W.PAPER_POT, precision=precision)
        if tune:
            h.autotune(3, 1.2, W.PAPER_MIX, 5)
        h.sweep(60, 1.2, W.PAPER_MIX, 5)
        h.sync()
        got.append({k: v for k, v in h.stats()[0].items() if k != "e_run"})
        h.close()
    assert got[0] == got[1]
