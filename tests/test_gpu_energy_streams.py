"""Energies of one unchanged state may overlap on the GPU: mc_energy_device only
enqueues, the handle's stream can be changed after it (nothing orders the two
streams), and a captured call can be replayed beside others.  Every one of them
gives the energy, and so does what the handle computes afterwards."""
import numpy as np
import pytest

from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _handle(Ms, seed=6):
    Ls = np.array([W.box_length(M) for M in Ms])
    st = [W.lattice_start(M, L, seed + k, candidates=8, passes=1) for k, (M, L) in enumerate(zip(Ms, Ls))]
    one = len(Ms) == 1
    h = F.Handle(float(Ls[0]) if one else Ls, np.concatenate([s[0] for s in st]), np.concatenate([s[1] for s in st]),
                 W.PAPER_POT, n_mol=None if one else np.array(Ms))
    h.sweep(5, 1.5, W.PAPER_MIX, 3)
    h.sync()
    return h


@pytest.mark.parametrize("Ms", [[8000], [64, 1000, 3000]])
def test_energies_on_two_streams(Ms):
    import torch
    h = _handle(Ms)
    E, P = h.energy(), h.pressure(1.0)
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs = torch.zeros((40, len(Ms)), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    for k in range(0, 40, 2):
        for j, s in enumerate(streams):
            h.set_stream(s.cuda_stream)
            h.energy_device(outs[k + j].data_ptr())
        assert np.array_equal(h.energy(), E)
    torch.cuda.synchronize()
    assert np.array_equal(outs.cpu().numpy(), np.broadcast_to(E, (40, len(Ms))))
    # the handle is as it was: later energies, virials and drift-free MD starts
    assert np.array_equal(h.energy(), E) and np.array_equal(h.pressure(1.0), P)
    h.close()


def test_replayed_energies_overlap():
    import torch
    h = _handle([3000])
    E = h.energy()[0]
    streams = [torch.cuda.Stream() for _ in range(2)]
    outs = [torch.zeros(1, dtype=torch.float64, device="cuda") for _ in streams]
    graphs = []
    for s, o in zip(streams, outs):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            h.set_stream(s.cuda_stream)
            for _ in range(4):
                h.energy_device(o.data_ptr())
        graphs.append(g)
    h.set_stream(0)
    torch.cuda.synchronize()
    for _ in range(20):
        for s, g, o in zip(streams, graphs, outs):
            with torch.cuda.stream(s):
                o.zero_()
                g.replay()
        assert h.energy()[0] == E
        torch.cuda.synchronize()
        assert [float(o[0]) for o in outs] == [E, E]
    h.close()
