"""The pair walks behind the energy, the virial and the MD forces where they
split: cells of more than 32 atoms, neighbourhoods of more than 192, two cells
per axis (each neighbour cell once), rows that wrap around the box, atoms with
more partners than a hit list or a contribution list holds; and a replica's
sums are the same alone and in a batch."""
import numpy as np
import pytest

import oracle
from oracle import md as OMD
from oracle import structure as OS
from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu

FAT = (1.5, 1.6, 1.7, 1.0, 33.75, 1.5)     # about 40 atoms inside a cutoff


def _handle(M, pot, n_cells=0, seed=3, sweeps=40):
    L = W.box_length(M)
    xyz, t = W.lattice_start(M, L, seed)
    h = F.Handle(L, xyz, t, pot, n_cells=n_cells)
    h.sweep(sweeps, 2.0, W.PAPER_MIX, seed)
    return h, L


CASES = [(64, W.PAPER_POT, 0), (216, W.PAPER_POT, 2), (300, W.PAPER_POT, 4), (512, W.PAPER_POT, 6), (125, FAT, 0),
         (343, FAT, 0)]


@pytest.mark.parametrize("M,pot,n_cells", CASES)
def test_energy_and_virial(M, pot, n_cells):
    h, L = _handle(M, pot, n_cells)
    q, _, t = h.state_fixed()
    assert h.energy()[0] == pytest.approx(oracle.energy(L, q, t, pot), rel=1e-12)
    assert h.pressure(1.0)[0, 0] == pytest.approx(OS.virial(L, q, t, pot), rel=1e-12)
    h.close()


@pytest.mark.parametrize("M,pot,n_cells", CASES)
@pytest.mark.parametrize("forces", ["fp64", "fp32"])
def test_forces(M, pot, n_cells, forces):
    h, L = _handle(M, pot, n_cells)
    q, _, t = h.state_fixed()
    f = OMD.forces(L, q, t, pot)
    # from rest, with a step in which nothing moves a quantum: v = dt F
    dt = 2.0 ** -40
    h.md_setup(dt, 0.0, 1.0, np.zeros((3 * M, 3)), forces)
    h.md_run(1)
    assert np.array_equal(h.state_fixed()[0], q)
    got = h.md_state()[0] / dt
    # a unit of 2^-53 (or 2^-24) in r^2 is up to 13 in a pair's force, which may
    # cancel against others': relative to the largest component
    tol = (64 * 13 * 2.0 ** -53 if forces == "fp64" else 64 * 13 * 2.0 ** -24) * np.abs(f).max()
    assert np.abs(got - f).max() <= tol
    h.close()


def test_a_replicas_sums_are_the_same_alone_and_in_a_batch():
    Ms, Ts = [64, 300, 27, 1000], [1.2, 2.0, 1.5, 0.9]
    Ls = [W.box_length(m) for m in Ms]
    st = [W.lattice_start(m, l, 20 + k) for k, (m, l) in enumerate(zip(Ms, Ls))]
    v0 = [W.maxwell_velocities(3 * m, T, 30 + k) for k, (m, T) in enumerate(zip(Ms, Ts))]
    hb = F.Handle(np.array(Ls), np.concatenate([s[0] for s in st]), np.concatenate([s[1] for s in st]), W.PAPER_POT,
                  n_mol=np.array(Ms))
    Eb, Pb = hb.energy(), hb.pressure(1.0)
    hb.md_setup(0.001, 1.0, np.array(Ts), np.concatenate(v0), "fp64")
    hb.md_run(11)                                        # one graph of eight steps and three of one
    vb, sb = hb.md_state()
    off = 0
    for k, M in enumerate(Ms):
        h = F.Handle(Ls[k], st[k][0], st[k][1], W.PAPER_POT)
        assert h.energy()[0] == Eb[k] and h.pressure(1.0)[0, 0] == Pb[k, 0]
        h.md_setup(0.001, 1.0, Ts[k], v0[k], "fp64")
        for n in (1, 8, 2):                              # split as no single call would
            h.md_run(n)
        v, s1 = h.md_state()
        assert np.array_equal(vb[off:off + 3 * M], v)
        assert sb[k, 2] == s1[0, 2] and sb[k, 3] == s1[0, 3]
        off += 3 * M
        h.close()
    hb.close()
