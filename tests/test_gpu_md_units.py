"""FP64 forces where a warp does not have one cell: dilute systems (several cells
to a warp, most of them empty, the last warp's cells fewer) and crowded cells
(several warps to a cell, cells with fewer and with more atoms than those take in
one go), against the oracle's forces; and a thermostatted run of such replicas is
the same alone and in a batch."""
import numpy as np
import pytest

from oracle import md as OMD
from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# (molecules, density, cells per axis asked for): 26^3 cells, four to a warp and two warps in the last block; 28^3, five to
# a warp and two cells in the last one; 48^3 or more, sixteen to a warp; eight cells of 129 and of 56 atoms; 14^3, one each
CASES = [(27, 0.0011, 0), (27, 0.00089, 0), (64, 0.0004, 0), (343, W.RHO, 2), (150, W.RHO, 2), (216, 0.05, 0)]


def _start(M, rho, seed):
    L = (3 * M / rho) ** (1.0 / 3.0)
    return L, W.lattice_start(M, L, seed, candidates=8, passes=1)


@pytest.mark.parametrize("M,rho,n_cells", CASES)
def test_forces(M, rho, n_cells):
    L, (xyz, t) = _start(M, rho, 3)
    h = F.Handle(L, xyz, t, W.PAPER_POT, n_cells=n_cells, warps_per_cell=2)
    h.sweep(20, 2.0, W.PAPER_MIX, 3)
    q, _, tt = h.state_fixed()
    f = OMD.forces(L, q, tt, W.PAPER_POT)
    dt = 2.0 ** -40                              # a step in which nothing moves a quantum: v = dt F
    h.md_setup(dt, 0.0, 1.0, np.zeros((3 * M, 3)), "fp64")
    h.md_run(1)
    assert np.array_equal(h.state_fixed()[0], q)
    got = h.md_state()[0] / dt
    # (as in the tests of the walk: a unit of 2^-53 in r^2 is up to 13 in a pair's force, which may cancel)
    assert np.abs(got - f).max() <= 64 * 13 * 2.0 ** -53 * np.abs(f).max()
    h.close()


def test_replicas_alone_and_in_a_batch():
    Ms = [27, 343, 64, 125]
    st = [_start(M, rho, 9) for M, rho in zip(Ms, (0.0011, W.RHO, 0.0004, W.RHO))]
    v0 = [W.maxwell_velocities(3 * M, 1.1, k) for k, M in enumerate(Ms)]

    def run(L, xyz, t, v, n_mol=None):
        h = F.Handle(L, xyz, t, W.PAPER_POT, n_mol=n_mol, n_cells=0, warps_per_cell=2)
        h.md_setup(0.001, 1.0, 1.1, v, "fp64")
        h.md_run(11)
        out = h.md_state()
        h.close()
        return out
    vb, sb = run(np.array([s[0] for s in st]), np.concatenate([s[1][0] for s in st]),
                 np.concatenate([s[1][1] for s in st]), np.concatenate(v0), np.array(Ms))
    off = 0
    for k, M in enumerate(Ms):
        v, s1 = run(st[k][0], st[k][1][0], st[k][1][1], v0[k])
        assert np.array_equal(vb[off:off + 3 * M], v) and sb[k, 2] == s1[0, 2] and sb[k, 3] == s1[0, 3]
        off += 3 * M
