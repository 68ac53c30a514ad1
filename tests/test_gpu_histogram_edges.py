"""The pair histogram where its FP32 placement cannot decide: distances exactly
on bin edges, the largest numbers of bins, and systems around a tile of 128
records.  Counts equal the oracle's, bin for bin."""
import numpy as np
import pytest

from oracle import structure as OS
from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _grid_molecules(m, L):
    """Right triangles with legs 1 on an m^3 lattice of spacing 2: every
    distance is the root of an integer, exact in the fixed-point box."""
    i = np.arange(m ** 3)
    corner = 2.0 * np.stack([i % m, (i // m) % m, i // (m * m)], axis=1)
    tri = np.array([[0.0, 0, 0], [1.0, 0, 0], [0, 1.0, 0]])
    xyz = (corner[:, None] + tri[None]).reshape(-1, 3)
    return xyz, np.tile(np.array([0, 1, 2], dtype=np.int32), m ** 3)


@pytest.mark.parametrize("dr,n_bins", [(0.25, 16), (1.0, 4), (0.125, 31), (1.0 / 3.0, 12)])
def test_distances_on_the_bin_edges(dr, n_bins):
    L = 8.0
    xyz, t = _grid_molecules(4, L)
    h = F.Handle(L, xyz, t, W.PAPER_POT)
    q, _, _ = h.state_fixed()
    counts, _ = h.pair_histogram(dr, n_bins)
    assert np.array_equal(counts[0].astype(np.int64), OS.pair_histogram(L, q, dr, n_bins))
    h.close()


@pytest.mark.parametrize("M", [42, 43, 64, 85, 86, 171])       # 126, 129, 192, 255, 258 and 513 records
@pytest.mark.parametrize("n_bins", [1, 7, 1024, 1025, 4096])   # four copies up to 1024, one above
def test_tiles_and_bin_counts(M, n_bins):
    L = W.box_length(M)
    xyz, t = W.lattice_start(M, L, M)
    h = F.Handle(L, xyz, t, W.PAPER_POT)
    h.sweep(20, 2.0, W.PAPER_MIX, M)
    q, _, _ = h.state_fixed()
    for dr in (0.5 * L / n_bins * (1.0 - 1e-9), 1e-3 * L / n_bins, 1e-12):
        counts, _ = h.pair_histogram(dr, n_bins)
        assert np.array_equal(counts[0].astype(np.int64), OS.pair_histogram(L, q, dr, n_bins)), dr
    h.close()
