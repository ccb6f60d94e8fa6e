"""The adjoint's sweeps at the edges of their tiles (16 x 12, 16 x 8, 8 x 12
and 8 x 4 faces): exactly one tile, one face more, the smallest grid, and grids
with rows that no face of the last tile has.  FP64 against the oracle's tangent
run: <lambda, v> = <r, dQ>, both exact derivatives, equal to rounding (1e-11 of
sums of up to 1e4 terms, as elsewhere).  FP32 against FP64 at 1e-5, as
elsewhere for weights without kinks."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2005_08736_gb300 import inputs  # noqa: E402
from paper_2005_08736_gb300.solver import Config, Simulation  # noqa: E402

GRIDS = [(6, 6, 6), (16, 12, 8), (17, 13, 9), (9, 25, 17), (33, 7, 13)]
DT = 0.05


def setup(n, recon, flux, prec):
    cfg = Config(*n, prec=prec, recon=recon, flux=flux, mu_ref=5e-3, p_ref=1.0, prandtl=0.7, visc=1, T_ref=1.0,
                 visc_exp=0.76)
    prim = inputs.random_smooth(n, seed=21, amp=0.15, kmax=1)
    q0 = torch.from_numpy(np.ascontiguousarray(oracle.conservative(prim, 1.4))).cuda()
    g = torch.Generator(device="cuda").manual_seed(13)
    r = torch.randn(cfg.shape, dtype=torch.float64, device="cuda", generator=g)
    v = torch.randn(cfg.shape, dtype=torch.float64, device="cuda", generator=g)
    return cfg, q0, r, v * q0.abs().amax(dim=(1, 2, 3), keepdim=True)


def gradient(cfg, q0, r):
    sim = Simulation(cfg)
    sim.init_conservative(q0)
    out = torch.empty_like(r)
    sim.adjoint_step(DT, r, out)
    torch.cuda.synchronize()
    sim.close()
    return out


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("recon,flux", [(0, 0), (1, 0), (1, 1)])
def test_fp64_adjoint_at_tile_edges(n, recon, flux):
    cfg, q0, r, v = setup(n, recon, flux, 0)
    grad = gradient(cfg, q0, r)
    t = oracle.TangentSolver(oracle.Config(*n, recon=recon, flux=flux, tau_num_C=0.0, prandtl=cfg.prandtl,
                                           visc_law=cfg.visc, mu_ref=cfg.mu_ref, T_ref=cfg.T_ref,
                                           visc_exp=cfg.visc_exp))
    t.set_state(q0.cpu().numpy(), v.cpu().numpy())
    t.step(1, DT)
    tan = float((r.cpu().numpy() * t.tangent()).sum())
    ad = (grad * v).sum().item()
    assert abs(ad - tan) <= 1e-11 * abs(tan), (ad, tan)


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("recon,flux", [(0, 0), (1, 0), (1, 1)])
def test_fp32_adjoint_at_tile_edges(n, recon, flux):
    grads = [gradient(cfg, q0, r) for cfg, q0, r, _ in (setup(n, recon, flux, p) for p in (0, 1))]
    err = ((grads[1] - grads[0]).abs().amax() / grads[0].abs().amax()).item()
    assert err <= 1e-5, err
