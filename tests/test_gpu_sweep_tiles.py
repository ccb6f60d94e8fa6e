"""Sweep kernels at the edges of their tiles against the FP64 oracle.

Grids one face past a tile (16 x 8 faces of k_sweep, 16 x 16 in FP64 with the smooth flux; 32 faces
by 10 layers of k_march), exactly one tile, the smallest grid the library
takes, and a walled direction, whose face n is a face of its own (in periodic
directions it is a copy of face 0).  Bounds as elsewhere: 1e-12 in FP64; 2e-5
in FP32 (fluxes rounded to 6e-8, divergences of the enthalpy flux amplified by
at most 1e2, a few steps).
"""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2005_08736_gb300 import inputs  # noqa: E402
from paper_2005_08736_gb300.solver import Config, Simulation  # noqa: E402

TOL = {0: 1e-12, 1: 2e-5}
# (recon, flux, characteristic variables)
KERNELS = [(0, 0, 0), (1, 0, 0), (2, 0, 1), (2, 1, 0), (1, 1, 1), (0, 1, 0)]
GRIDS = [(6, 6, 6), (16, 8, 10), (17, 9, 11), (11, 33, 17), (33, 11, 9)]


def check(cfg, prim):
    sim = Simulation(cfg)
    sim.init_primitive(prim)
    sim.step(2)
    got = sim.state()
    sim.close()
    c = cfg
    o = oracle.Solver(oracle.Config(c.nx, c.ny, c.nz, lx=c.lx, ly=c.ly, lz=c.lz, y0=c.y0, y_stretch=c.y_stretch,
                                    stretch_b=c.stretch_b, bc_y=c.bc_y, gamma=c.gamma, prandtl=c.prandtl,
                                    visc_law=c.visc, mu_ref=c.mu_ref, T_ref=c.T_ref, visc_exp=c.visc_exp,
                                    T_wall=c.T_wall, recon=c.recon, flux=c.flux, tau_num_C=c.tau_num_C, cfl=c.cfl,
                                    char_recon=c.recon_vars))
    o.set_state(oracle.conservative(prim, c.gamma))
    o.step(2)
    ref = o.state()
    scale = [np.abs(ref[v]).max() for v in range(5)]
    scale[1:4] = [max(scale[1:4])] * 3
    err = max(np.abs(got[v] - ref[v]).max() / scale[v] for v in range(5))
    assert err <= TOL[cfg.prec], err


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("recon,flux,char", KERNELS)
def test_periodic_grid_at_tile_edges(recon, flux, char, n, prec):
    cfg = Config(*n, prec=prec, recon=recon, flux=flux, recon_vars=char, tau_num_C=1.0, mu_ref=5e-3, p_ref=1.0,
                 prandtl=0.7, visc=1, T_ref=1.0, visc_exp=0.76)
    check(cfg, inputs.random_smooth(n, seed=41, amp=0.15, kmax=1))


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("recon,flux,char", KERNELS)
def test_walled_stretched_grid(recon, flux, char, prec):
    n = (17, 20, 9)
    cfg = Config(*n, lx=2 * math.pi, ly=2.0, y0=-1.0, lz=math.pi, y_stretch=1, stretch_b=2.0, bc_y=1, T_wall=1.0,
                 prec=prec, recon=recon, flux=flux, recon_vars=char, tau_num_C=1.0, mu_ref=5e-3, p_ref=1.0)
    check(cfg, inputs.random_smooth(n, seed=42, amp=0.1, kmax=1))
