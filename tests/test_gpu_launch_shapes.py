"""Launch shapes of the sweeps: what earlier builds stored is accepted and does
not slow the step down, and members that differ in it share batched launches."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2005_08736_gb300 import inputs  # noqa: E402
from paper_2005_08736_gb300.solver import Config, Ensemble, Simulation, taylor_green_config  # noqa: E402


def simulation(n, shape=(0, 0)):
    sim = Simulation(taylor_green_config(n, "fp32"))
    sim._call(sim.lib.hgks_set_sweep_shape(sim.h, *shape))
    sim.init_primitive(inputs.taylor_green(n))
    return sim


def sweep_ms(*sims):
    """Shortest stage-1 sweeps of each simulation, taken in turn after warm-up."""
    for sim in sims:
        sim.step(20, 1e-5)
    best = [1e30] * len(sims)
    for _ in range(8):
        for k, sim in enumerate(sims):
            best[k] = min(best[k], sim.profile_step(1e-5)["flux_stage1"])
    return best


@pytest.mark.parametrize("shape", [(3, 16), (0, 64), (1, 8), (0, 2 ** 31 - 1)])
def test_stored_shapes_cost_no_more_than_the_automatic_one(shape):
    # 64^3: 64 rows a block made the sweeps 2.5 times as long, 8 rows 1.2 times;
    # two runs of one shape differ by a few per cent.
    stored, automatic = sweep_ms(simulation(64, shape), simulation(64))
    assert stored <= 1.1 * automatic, (stored, automatic)


@pytest.mark.parametrize("n", [(6, 6, 256), (6, 256, 6), (256, 6, 6), (16, 16, 200)])
def test_long_boxes_are_split_evenly(n):
    # One layer per CTA is the shortest march; the automatic split may be
    # longer where that saves start-ups, never much slower.  The long axis's
    # few tiles once marched up to 18 layers each: 1.3 to 2.7 times as long.
    sims = []
    for chunk in (0, 1):
        sim = Simulation(Config(*n, prec=1, recon=2, flux=1, tau_num_C=1.0, mu_ref=5e-3, p_ref=1.0))
        sim._call(sim.lib.hgks_set_sweep_shape(sim.h, 0, chunk))
        sim.init_primitive(inputs.random_smooth(n, seed=3, amp=0.1, kmax=1))
        sims.append(sim)
    automatic, single = sweep_ms(*sims)
    assert automatic <= 1.15 * single, (automatic, single)


def test_members_with_other_stored_shapes_share_batched_launches():
    ens = Ensemble([simulation(16), simulation(16, (3, 16))], batched=True)
    ens.step(2)
    a, b = (s.state(device=True) for s in ens.sims)
    assert torch.equal(a, b)
    ens.close()


@pytest.mark.parametrize("batched", [True, False])
def test_members_of_an_ensemble_share_the_chip(batched):
    # 24 boxes of 32^3 against one box of as many cells: 1.6 times as long
    # (1.4 as branches); with every member split over all SMs 2.1 (1.9) times.
    n = (64, 96, 128)
    one = Simulation(Config(*n, prec=1))
    one.init_primitive(inputs.random_smooth(n, seed=1, amp=0.05, p0=100 / 1.4))
    ens = Ensemble([simulation(32) for _ in range(24)], batched=batched)
    runs = [(ens.step, ens.sims[0].stream), (one.step, one.stream)]
    best = [1e30, 1e30]
    for _ in range(8):
        for k, (step, stream) in enumerate(runs):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            step(4, 1e-4, sync=False)
            a.record(stream)
            step(4, 1e-4, sync=False)
            b.record(stream)
            torch.cuda.synchronize()
            best[k] = min(best[k], a.elapsed_time(b))
    ens.close()
    assert best[0] <= 1.8 * best[1], best
