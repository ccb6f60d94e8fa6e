"""A device state read while the current stream still converts an earlier one
leaves that conversion alone (see test_state_ordering.py for the order)."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2005_08736_gb300 import inputs  # noqa: E402
from paper_2005_08736_gb300.solver import Config, Simulation  # noqa: E402


def test_states_read_one_after_another_do_not_overwrite_each_other():
    sims = []
    for k in range(2):
        sim = Simulation(Config(16, 16, 16, prec=0, p_ref=1.0))
        sim.init_primitive(inputs.random_smooth((16, 16, 16), seed=k, amp=0.1))
        sims.append(sim)
    want = [s.state() for s in sims]
    first = sims[0].state(device=True)
    torch.cuda._sleep(20_000_000)  # some 10 ms of work before the conversion
    converted = first.to(torch.float32)
    del first
    sims[0].stream.synchronize()
    second = sims[1].state(device=True)
    torch.cuda.synchronize()
    assert torch.equal(converted.cpu(), torch.from_numpy(want[0]).float())
    assert torch.equal(second.cpu(), torch.from_numpy(want[1]))


def test_the_default_stream_stands_for_a_stream_of_its_own():
    # The library cannot capture the default stream and takes one of its own
    # for it; the tensors' order follows the stream the simulation knows.
    cfg = Config(16, 16, 16, prec=0, p_ref=1.0)
    prim = torch.from_numpy(inputs.random_smooth((16, 16, 16), seed=3, amp=0.1))
    ref = Simulation(cfg)
    ref.init_primitive(prim)
    sim = Simulation(cfg, stream=torch.cuda.default_stream())
    assert sim.stream.cuda_stream != 0
    torch.cuda._sleep(20_000_000)
    sim.init_primitive(prim.cuda(non_blocking=True))
    sim.step(2, 1e-3, sync=False)
    got = sim.state(device=True)
    ref.step(2, 1e-3)
    assert torch.equal(got.cpu(), torch.from_numpy(ref.state()))
