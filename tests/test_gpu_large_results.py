"""Results whose size is the caller's choice (wavevectors or bins times the
replicas): several batches of wavevectors and a result beyond what the handle
keeps give the values of small calls, and a large call's workspace is given back."""
import numpy as np
import pytest

from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu

R, M = 256, 27


@pytest.fixture(scope="module")
def handle():
    L = W.box_length(M)
    st = [W.lattice_start(M, L, k, candidates=4, passes=1) for k in range(R)]
    h = F.Handle(np.full(R, L), np.concatenate([s[0] for s in st]), np.concatenate([s[1] for s in st]), W.PAPER_POT,
                 n_mol=np.full(R, M, dtype=np.int32))
    yield h, L
    h.close()


def test_structure_factor_in_batches(handle):
    import torch
    h, L = handle
    n_q = 40000                                  # 82 MB of results, in batches of 1024 wavevectors
    q = 2 * np.pi / L * np.random.default_rng(4).integers(-9, 10, (n_q, 3)).astype(np.float64)
    h.structure_factor(q[:64])
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    S = h.structure_factor(q)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= 64 << 20
    for k in (0, 777, 13107, 39000):
        assert np.array_equal(S[:, k:k + 1000], h.structure_factor(q[k:k + 1000]))


def test_histogram_of_many_replicas(handle):
    h, L = handle
    n = 4096
    dr = 0.5 * L / n * (1 - 1e-9)
    counts, g = h.pair_histogram(dr, n)
    coarse, _ = h.pair_histogram(8 * dr, n // 8)
    # (a bin edge of the coarse histogram is one of the fine one's up to rounding: pairs that near an edge are rare)
    diff = np.abs(counts.reshape(R, n // 8, 8).sum(axis=2).astype(np.int64) - coarse.astype(np.int64))
    assert diff.sum() <= 2
    assert np.isfinite(g).all()
