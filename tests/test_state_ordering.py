"""Stream order of Simulation.state(device=True) (CPU only, stand-ins for the
stream, the allocator and the library): the tensor's memory belongs to the
current stream, where work queued earlier may still read what was freed to make
it, so the library has to write it on that stream.  Written on the simulation's
own stream instead, a state read right after another one could overwrite the
other while it was still being converted (an ensemble's members, read in a
loop)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2005_08736_gb300.solver import Config, Simulation  # noqa: E402


class Stream:
    def __init__(self, handle):
        self.cuda_stream = handle


class Tensor:
    def __init__(self, owner):
        self.owner = owner

    def data_ptr(self):
        return 64


def test_device_state_is_written_on_the_stream_that_owns_its_memory(monkeypatch):
    current, own = Stream(11), Stream(22)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: current)
    monkeypatch.setattr(torch, "empty", lambda *a, **k: Tensor(current.cuda_stream))
    calls = []

    class Lib:
        def hgks_get_state_on(self, h, p, stream):
            calls.append((p.value, stream.value))
            return 0

    sim = object.__new__(Simulation)
    sim.lib, sim.h, sim.cfg, sim.device, sim.stream = Lib(), None, Config(8, 8, 8), None, own
    out = sim.state(device=True)
    assert out.owner == 11 and calls == [(64, 11)]
