"""A read-out whose wait fails.  The failure is made on the host: the handle's
stream is being captured, and a stream under capture cannot be waited for (the
call returns an error; nothing runs on the GPU).  The handle works as before on
its own stream."""
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
