"""Walled FP32 runs repeat bit for bit, whatever ran on the GPU before.

With walls and an even number of cells in y the last pair of face layers of
k_march is (face n, face n + 1), the second of which does not exist; nothing
that other launches left in shared memory may decide how face n is evaluated.
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from paper_2005_08736_gb300 import inputs  # noqa: E402
from paper_2005_08736_gb300.solver import Config, Simulation  # noqa: E402


def run(n, seed, wall, steps, recon=0, flux=0, p0=1.0, amp=0.05):
    kw = dict(ly=2.0, y0=-1.0, y_stretch=1, stretch_b=2.0, bc_y=1, T_wall=1.0) if wall else {}
    cfg = Config(*n, lx=2 * math.pi, lz=math.pi, prec=1, recon=recon, flux=flux, tau_num_C=1.0, mu_ref=5e-3,
                 p_ref=p0, **kw)
    sim = Simulation(cfg)
    sim.init_primitive(inputs.random_smooth(n, seed=seed, amp=amp, kmax=1, p0=p0))
    sim.step(steps, 1e-3)
    out = sim.state()
    sim.close()
    return out


@pytest.mark.parametrize("n", [(40, 20, 17), (33, 16, 12), (64, 36, 24)])
def test_walled_run_repeats_after_other_runs(n):
    # A nearly uniform state: next to leftover zeros (a uniform run before) every jump is below the limit
    # of the compatibility state's midpoint rule, next to leftover data of size 1e5 it is not.
    out = []
    for before in (dict(amp=0.0), dict(amp=0.5, p0=1e6), dict(amp=0.0), dict(amp=0.5, recon=2, flux=1)):
        run((64, 64, 64), 7, False, 1, **before)
        out.append(run(n, 1, True, 3, amp=0.005))
    for later in out[1:]:
        assert np.array_equal(later, out[0])
