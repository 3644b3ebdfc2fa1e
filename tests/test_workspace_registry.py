"""The workspace registry of the binding against a stand-in for the library and for two devices (no GPU needed).

The library files one workspace address per device and goes on using it; the binding owns the memory.  So the memory behind an
address must live as long as the address is registered, whatever happens on the other devices in between."""
import gc
import weakref

import pytest
import torch

from paper_2508_20407_b200 import binding as tl


class Buffer:
    """What the registry reads of a CUDA tensor."""
    is_cuda = True

    def __init__(self, nbytes, device):
        self.nbytes, self.device = nbytes, torch.device(device)

    def is_contiguous(self):
        return True

    def numel(self):
        return self.nbytes

    def element_size(self):
        return 1

    def data_ptr(self):
        return id(self)


class Machine:
    """Two devices, each with the address that the library holds for it, and every buffer that was ever handed out."""

    def __init__(self):
        self.current, self.registered, self.alive = 0, {}, {}

    def lib(self):
        return self

    def tlin_set_workspace(self, ptr, nbytes):
        self.registered[self.current] = ptr
        return tl.TLIN_OK

    def empty(self, nbytes, dtype=None, device=None):
        device = torch.device(device)
        b = Buffer(nbytes, torch.device("cuda", self.current) if device.index is None else device)
        self.alive[id(b)] = weakref.ref(b)
        return b

    def check(self):
        """Every registered address belongs to a buffer that still exists and lies on that device."""
        gc.collect()
        for device, ptr in self.registered.items():
            if ptr is not None:
                b = self.alive[ptr]()
                assert b is not None, f"the library's workspace of device {device} has been freed"
                assert b.device.index == device


@pytest.fixture
def machine(monkeypatch):
    m = Machine()
    monkeypatch.setattr(tl, "lib", m.lib)
    monkeypatch.setattr(tl, "_current_device", lambda: m.current)
    monkeypatch.setattr(tl, "_workspaces", {}, raising=False)
    monkeypatch.setattr(tl, "_workspace_sizes", {}, raising=False)
    monkeypatch.setattr(tl, "_workspace_tensor", None)
    monkeypatch.setattr(torch, "empty", m.empty)
    return m


def on(m, device, nbytes):
    m.current = device
    t = tl.ensure_workspace(nbytes, torch.device("cuda", device))
    assert t is None or (t.device.index == device and t.numel() >= nbytes)
    m.check()
    return t


def test_a_device_keeps_its_workspace_while_another_one_gets_its_own(machine):
    first = on(machine, 0, 5 << 20)
    on(machine, 1, 9 << 20)                        # layers on device 0, then on device 1: the forward pass of a split model
    machine.current = 0                            # its backward pass uses what the library has for device 0, unasked
    assert machine.registered[0] == first.data_ptr()
    machine.check()
    assert on(machine, 0, 5 << 20) is first        # and nothing is allocated again on the way back and forth
    assert on(machine, 1, 9 << 20).device.index == 1
    assert len(machine.alive) == 2


def test_growing_and_dropping_touch_the_current_device_only(machine):
    small = on(machine, 0, 1 << 20)
    other = on(machine, 1, 1 << 20)
    ref = weakref.ref(small)
    del small
    large = on(machine, 0, 4 << 20)
    gc.collect()
    assert ref() is None                           # the replaced buffer is given back
    assert machine.registered == {0: large.data_ptr(), 1: other.data_ptr()}
    machine.current = 1
    tl.set_workspace(None)
    machine.check()
    assert machine.registered == {0: large.data_ptr(), 1: None}
    assert on(machine, 1, 0) is None
    assert on(machine, 0, 4 << 20) is large


def test_a_buffer_of_another_device_is_replaced(machine):
    machine.current = 1
    tl.set_workspace(machine.empty(8 << 20, device="cuda:0"))       # registered for device 1 by mistake
    assert on(machine, 1, 1 << 20).device.index == 1
    assert tl.ensure_workspace(1 << 20, "cuda") is tl._workspaces[1]


def test_the_callers_own_buffer_is_used_as_it_is(machine):
    mine = machine.empty(3 << 20, device="cuda:0")
    tl.set_workspace(mine)
    assert on(machine, 0, 3 << 20) is mine and tl._workspace_tensor is mine
    assert on(machine, 0, (3 << 20) + 1) is not mine
