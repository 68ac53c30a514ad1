"""What reads the cell list directly after mc_autotune (its trial sweeps rebuild
the list, and nothing rebuilds it before the next sweep): energy, virial and the
first MD steps are those without the call, bit for bit."""
import numpy as np
import pytest

from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Ms", [[64], [1000], [64, 300, 125]])
@pytest.mark.parametrize("forces", ["fp64", "fp32"])
def test_cell_list_after_autotune(Ms, forces):
    one = len(Ms) == 1
    Ls = np.array([W.box_length(M) for M in Ms])
    st = [W.lattice_start(M, L, 50 + k) for k, (M, L) in enumerate(zip(Ms, Ls))]
    seeds = 5 if one else np.arange(len(Ms), dtype=np.uint64)
    v0 = W.maxwell_velocities(3 * int(np.sum(Ms)), 1.4, 7)
    got = []
    for tune in (True, False):
        h = F.Handle(float(Ls[0]) if one else Ls, np.concatenate([s[0] for s in st]), np.concatenate([s[1] for s in st]),
                     W.PAPER_POT, n_mol=None if one else np.array(Ms))
        h.sweep(7, 1.4, W.PAPER_MIX, seeds)
        if tune:
            h.autotune(3, 1.4, W.PAPER_MIX, seeds)
        out = [h.energy(), h.pressure(1.4)]
        h.md_setup(0.001, 1.0, 1.4, v0, forces)
        h.md_run(2)
        out += list(h.md_state()) + list(h.state_fixed())
        got.append(out)
        h.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
