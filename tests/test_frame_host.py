"""Host logic of a frame's binning: what is queued behind the binning before its status is read is
waited for when the binning failed, before the workspace that it reads is given up."""
import ctypes
from types import SimpleNamespace

import pytest
import torch

from paper_2308_04079_gb300 import _abi as abi
from paper_2308_04079_gb300 import rasterizer


class _Status:
    """A frame whose binning reports the given status flags, one per attempt, and a log of the order
    of launches, waits, and workspaces taken."""

    def __init__(self, monkeypatch, flags):
        self.log = log = []
        nbytes = ctypes.sizeof(abi.gs_device_status)
        attempts = iter(flags)
        fr = self.frame = rasterizer.Frame.__new__(rasterizer.Frame)
        fr.layout = SimpleNamespace(status=0)
        fr.ws = torch.zeros(nbytes, dtype=torch.uint8)

        def bin_sort():
            st = abi.gs_device_status()
            st.flags, st.num_instances = next(attempts), 1000
            fr.ws.copy_(torch.frombuffer(bytearray(bytes(st)), dtype=torch.uint8))
            log.append("bin")

        fr.preprocess = lambda g: None
        fr.bin_sort = bin_sort
        fr._alloc = lambda capacity: log.append("workspace")
        fr._host_status = (torch.zeros(nbytes, dtype=torch.uint8),
                           SimpleNamespace(record=lambda: None, synchronize=lambda: log.append("status")))
        stream = SimpleNamespace(synchronize=lambda: log.append("wait"))
        monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: stream)

    def run(self):
        self.frame._binned_then(None, lambda: self.log.append("blend"))


def test_the_old_workspace_is_given_up_after_the_blend_queued_on_it(monkeypatch):
    s = _Status(monkeypatch, [abi.FLAG_CAPACITY, 0])
    s.run()
    assert s.log == ["bin", "blend", "status", "wait", "workspace", "bin", "blend", "status"]
    assert s.frame.last_status.num_instances == 1000


@pytest.mark.parametrize("flag", [abi.FLAG_TIMEOUT, abi.FLAG_INTERNAL])
def test_nothing_is_in_flight_when_a_failed_binning_is_raised(monkeypatch, flag):
    s = _Status(monkeypatch, [flag])
    with pytest.raises(abi.GSError):
        s.run()
    assert s.log == ["bin", "blend", "status", "wait"]


def test_a_binning_that_succeeds_is_not_waited_for_beyond_its_status(monkeypatch):
    s = _Status(monkeypatch, [0])
    s.run()
    assert s.log == ["bin", "blend", "status"]


class _Device(torch.Tensor):
    """A host tensor that passes for a device tensor where only its attributes are looked at."""
    is_cuda = True


def _tensors(n=3):
    def t(*shape):
        return torch.rand(*shape).as_subclass(_Device)
    return rasterizer.GaussianTensors(t(n, 3), t(n, 3), t(n, 4), t(n), t(n, 4, 3), 1)


FIELDS = ("means", "scales", "quats", "opacities", "sh")


def test_prepared_tensors_are_not_the_callers_own():
    """prepared() is kept across calls (a batch's Gaussians, a forward pass's inputs until its backward
    pass): it shares the caller's values, but not what becomes of the caller's tensor objects."""
    g = _tensors()
    p = g.prepared()
    want = {k: (getattr(p, k).data_ptr(), getattr(p, k).shape) for k in FIELDS}
    for k in FIELDS:
        t = getattr(g, k)
        assert t.data_ptr() == want[k][0]
        t[0] = 2.0                                       # a new value is seen
        assert torch.all(getattr(p, k)[0] == 2.0)
        old = t.detach()
        t.data = torch.zeros(1).as_subclass(_Device)     # another tensor in its place is not
        assert (getattr(p, k).data_ptr(), getattr(p, k).shape) == want[k] == (old.data_ptr(), old.shape)
        getattr(p, k).requires_grad_()
        assert not t.requires_grad
