"""Cosines of fixed-point displacements in integer arithmetic (correlations and
S(q)): wavevectors off the box lattice, far beyond it and not finite,
displacements of several boxes, list lengths around the eight slices of a
block, and replicas that end inside a block of 32 molecules."""
import numpy as np
import pytest

from oracle import observables as OO
from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu

EPS = 2.0 ** -52


def _system(M, seed):
    L = W.box_length(M)
    xyz, t = W.lattice_start(M, L, seed)
    h = F.Handle(L, xyz, t, W.PAPER_POT)
    h.sweep(30, 2.0, W.PAPER_MIX, seed)
    return h, L


def _phases(L, q, qv):
    """q . x in extended precision, radians."""
    x = q.astype(np.longdouble) * (np.longdouble(L) / np.longdouble(2.0) ** 32)
    return (x[:, None, :] * qv.astype(np.longdouble)[None]).sum(axis=2)


@pytest.mark.parametrize("scale", [1e-3, 1.0, 7.4, 1e4, 1e8])
@pytest.mark.parametrize("M", [64, 1366])                     # 192 records; 4098: one part of 4096 and two
def test_structure_factor_of_any_wavevector(M, scale):
    h, L = _system(M, 3)
    qv = np.random.default_rng(5).normal(size=(7, 3)) * scale
    qv[0] = [scale, 0.0, -0.0]
    q, _, _ = h.state_fixed()
    n = 3 * M
    ph = _phases(L, q, qv)
    # what extended precision itself leaves in a phase of this size
    noise = float(np.abs(ph).max()) * float(np.finfo(np.longdouble).eps)
    rho = np.exp(-1j * 0) * (np.cos(ph).sum(axis=0).astype(float) + 1j * np.sin(ph).sum(axis=0).astype(float))
    # n cosines to a unit of 2^-53 each, and 2 |rho| times that in the square
    tol = 4.0 * (EPS + noise) * n * (np.abs(rho) + 1.0) / n + 8 * EPS * np.abs(rho) ** 2 / n
    assert np.all(np.abs(h.structure_factor(qv)[0] - np.abs(rho) ** 2 / n) <= tol)
    h.close()


def test_structure_factor_not_finite():
    h, L = _system(64, 3)
    qv = np.array([[np.nan, 0, 0], [1.0, 0, 0], [0, np.inf, 0], [0, 0, 0]])
    S = h.structure_factor(qv)[0]
    assert np.isnan(S[0]) and np.isnan(S[2]) and np.isfinite(S[1]) and S[3] == 192.0
    h.close()


@pytest.mark.parametrize("Ms", [[64], [33, 64, 31], [97, 13]])
@pytest.mark.parametrize("nqa,nqc", [(1, 1), (7, 9), (8, 16), (256, 3)])
def test_observables_across_boxes(Ms, nqa, nqc):
    Ls = np.array([W.box_length(max(M, 20)) for M in Ms])
    st = [W.lattice_start(M, L, 7 + k) for k, (M, L) in enumerate(zip(Ms, Ls))]
    one = len(Ms) == 1
    h = F.Handle(float(Ls[0]) if one else Ls, np.concatenate([s[0] for s in st]), np.concatenate([s[1] for s in st]),
                 W.PAPER_POT, n_mol=None if one else np.array(Ms))
    h.sweep(50, 1.5, W.PAPER_MIX, 4)
    q0, X0, t0 = h.state_fixed()
    h.set_t0()
    # a common drift carries every atom several boxes in 300 steps
    v = W.maxwell_velocities(h.N, 1.0, 3) + np.array([60.0, -45.0, 0.0])
    h.md_setup(0.001, 0.0, 1.0, v)
    h.md_run(300)
    q, X, _ = h.state_fixed()
    assert np.abs(X - X0).max() > 2 ** 33
    rng = np.random.default_rng(11)
    qa, qc = 7.4 * rng.normal(size=(nqa, 3)), 5.1 * rng.normal(size=(nqc, 3))
    out, fs, fcm, c2 = h.observables(qa, qc, per_particle=True)
    off = 0
    for k, M in enumerate(Ms):
        sl, sm = slice(off, off + 3 * M), slice(off // 3, off // 3 + M)
        kref = OO.reference_sites(t0[sl])
        o = OO.observables(Ls[k], X[sl], X0[sl], q[sl], OO.orientation(q0[sl], Ls[k], kref), kref, qa, qc)
        # the oracle's phases (up to 9 sigma of q times 25 sigma of drift) carry their size times 2^-52
        tol = 600.0 * 3 * EPS
        assert np.abs(fs[sl] - o["F_s_i"]).max() <= tol
        assert np.abs(fcm[sm] - o["F_s_cm_i"]).max() <= tol
        assert np.abs(c2[sm] - o["C_2_i"]).max() <= 64 * EPS
        assert np.abs(out[k] - [o["F_s"], o["F_s_cm"], o["C_2"]]).max() <= tol
        off += 3 * M
    qa[0, 1] = np.nan
    out2, fs2, fcm2, _ = h.observables(qa, qc, per_particle=True)
    assert np.isnan(fs2).all() and np.array_equal(fcm2, fcm) and np.isnan(out2[:, 0]).all()
    h.close()


def test_time_zero_is_exactly_one():
    h, L = _system(100, 6)
    h.set_t0()
    qa = 7.4 * np.random.default_rng(2).normal(size=(49, 3))
    out, fs, fcm, c2 = h.observables(qa, qa[:7], per_particle=True)
    assert (fs == 1.0).all() and (fcm == 1.0).all() and np.abs(c2 - 1.0).max() <= 8 * EPS
    assert out[0, 0] == 1.0 and out[0, 1] == 1.0
    h.close()
