"""A read-out whose wait fails hands over nothing.  The failure is made on the
host: the handle's stream is being captured, and a stream under capture cannot
be waited for (the call returns an error; nothing runs on the GPU).  The caller's
arrays stay as they were, and the handle works as before on its own stream."""
import numpy as np
import pytest

from paper_2506_21290_gb300 import flipmc as F
from paper_2506_21290_gb300 import workloads as W

pytestmark = pytest.mark.gpu


class _Capture:
    """A stream under capture for the length of a with block, whatever becomes of the capture."""

    def __enter__(self):
        import torch
        self.stream, self.graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        self._ctx = torch.cuda.stream(self.stream)
        self._ctx.__enter__()
        self.graph.capture_begin(capture_error_mode="relaxed")
        return self.stream.cuda_stream

    def __exit__(self, *exc):
        try:
            self.graph.capture_end()     # the failed wait has ended the capture
        except RuntimeError:
            pass
        self._ctx.__exit__(None, None, None)
        return False


def _reads(M, n_bins, n_q):
    N, mark = 3 * M, 12345.0
    q = np.random.default_rng(1).normal(size=(n_q, 3))

    def dbl(n):
        return np.full(n, mark)

    lib = F.load
    P = lambda a: a.ctypes.data   # noqa: E731
    stats = (F.mc_stats * 1)()
    stats[0].sweeps = 777
    T = np.array([1.0])
    E, pr, S, hist, g, v, out = dbl(1), dbl(2), dbl(n_q), np.full(n_bins, 777, dtype=np.uint64), dbl(n_bins), dbl(3 * N), dbl(5)
    xyz, types = dbl(3 * N), np.full(N, 77, dtype=np.int32)
    calls = {
        "energy": lambda h: lib().mc_energy(h, P(E)),
        "pressure": lambda h: lib().mc_pressure(h, P(T), P(pr)),
        "structure factor": lambda h: lib().mc_structure_factor(h, P(q), n_q, P(S)),
        "histogram": lambda h: lib().mc_pair_histogram(h, 0.01, n_bins, P(hist), P(g)),
        "md state": lambda h: lib().mc_md_state(h, P(v), P(out)),
        "statistics": lambda h: lib().mc_state(h, None, None, F.C.addressof(stats)),
        "state": lambda h: lib().mc_state(h, P(xyz), P(types), F.C.addressof(stats)),
    }

    def untouched():
        return (all((a == mark).all() for a in (E, pr, S, g, v, out, xyz)) and (hist == 777).all() and (types == 77).all()
                and stats[0].sweeps == 777 and stats[0].e_run == 0.0)
    return calls, untouched


def _handle(M):
    L = W.box_length(M)
    xyz, t = W.lattice_start(M, L, 3)
    h = F.Handle(L, xyz, t, W.PAPER_POT)
    h.md_setup(0.001, 1.0, 1.0, W.maxwell_velocities(3 * M, 1.0, 2), "fp64")
    h.md_run(3)
    return h


def test_the_call_after_a_failed_wait_works():
    h = _handle(125)
    E = h.energy()
    with _Capture() as stream:
        h.set_stream(stream)
        with pytest.raises(F.McError) as e:
            h.energy()
        assert e.value.code == F.MC_ERR_CUDA
    h.set_stream(0)
    assert np.array_equal(h.energy(), E)
    h.close()


def test_outputs_of_a_failed_wait_are_left_alone():
    import torch
    M = 125
    h = _handle(M)
    # (an earlier call's results are in the buffer that the failed calls would read)
    E, P, v = h.energy(), h.pressure(1.0), h.md_state()[0]
    calls, untouched = _reads(M, 50, 12)
    for name, call in calls.items():
        torch.cuda.synchronize()
        with _Capture() as stream:
            h.set_stream(stream)
            rc = call(h.h)
        h.set_stream(0)
        assert rc == F.MC_ERR_CUDA, (name, rc)
        assert untouched(), name
    assert np.array_equal(h.energy(), E) and np.array_equal(h.pressure(1.0), P) and np.array_equal(h.md_state()[0], v)
    h.close()
