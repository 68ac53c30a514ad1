"""MD steps and MC sweeps may alternate: the first step after sweeps, a logged or
timed sweep, or a new state begins with the forces of the configuration it
starts from, as a run set up there does; autotuning trials change nothing."""
import numpy as np
import pytest

from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _between(h, how, T):
    if how == "sweep":
        h.sweep(3, T, W.PAPER_MIX, 4)
    elif how == "logged":
        h.sweep_logged(2, T, W.PAPER_MIX, 4)
    elif how == "timed":
        h.sweep_timed(2, T, W.PAPER_MIX, 4)
    elif how == "autotune":
        h.autotune(2, T, W.PAPER_MIX, 4)
    elif how == "state":
        q, X, t = h.state_fixed()
        t = t.reshape(-1, 3)[:, [1, 0, 2]].reshape(-1).copy()      # another atom order in every molecule
        h.set_state_fixed(q, X, t)


@pytest.mark.parametrize("how", ["sweep", "logged", "timed", "autotune", "state"])
@pytest.mark.parametrize("forces", ["fp64", "fp32"])
def test_first_step_after_a_change(how, forces):
    M, T = 216, 1.5
    L = W.box_length(M)
    xyz, t = W.lattice_start(M, L, 11)
    h = F.Handle(L, xyz, t, W.PAPER_POT)
    h.sweep(50, T, W.PAPER_MIX, 11)
    h.md_setup(0.001, 0.0, T, W.maxwell_velocities(3 * M, T, 12), forces)
    h.md_run(5)
    v = h.md_state()[0]
    _between(h, how, T)
    q, X, tt = h.state_fixed()
    g = F.Handle(L, xyz, t, W.PAPER_POT)
    g.set_state_fixed(q, X, tt)
    g.md_setup(0.001, 0.0, T, v, forces)
    for k in (h, g):
        k.md_run(1)
    # (the two cell lists have different shifts, so a force may add its pairs in another order; one step of 1e-3 with
    # forces that are a configuration behind is off by more than 1e-3)
    a, b = h.md_state()[0], g.md_state()[0]
    tol = 1e-12 if forces == "fp64" else 1e-4
    assert np.abs(a - b).max() <= tol * max(1.0, np.abs(b).max())
    h.close()
    g.close()
