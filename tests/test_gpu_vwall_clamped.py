"""Velocity walls beside a BE cell clamped at z_c: its ghost is f^eq(n_wall, 0, theta_wall) +
f* - f^eq, f^eq the equilibrium of the cell's own n and eps at the force-shifted velocity,
as in the oracle, although the cell itself relaxes to the energy of the equilibrium at z_c.

A uniform state, halo included, is streamed onto itself, so one step relaxes the known
populations, and the stored ghost rows are compared with the oracle's equilibria, by the
step of few tiles and by the one-thread-per-cell step (a persistent grid of one block).
Tolerance: the oracle evaluates g_1(z_c) = -ln(1 - z_c) from the rounded z_c, off by up
to 2^-53 / (1 - z_c) = 1.1e-9, which enters f^eq times 2 pi theta Q_00 with theta = 1.2 and
Q_00 below 1: 1e-8."""
import numpy as np
import pytest

from paper_1709_09073_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [0, 1])
@pytest.mark.parametrize("accel", [(0.0, 0.0), (2e-3, -1e-3)])
def test_ghosts_of_clamped_cells(orc, grid, accel):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1709_09073_gb300 import build, rlbm as R
    build.build()
    R.load()
    nx, ny, tau, tw, nw = 5, 9, 0.9, 1.05, 1.1
    P, V = W.PERIODIC, W.VELOCITY_WALL
    f = 2.0 * orc.feq(W.BE, 0.95, 0.03, -0.02, 0.9)  # twice the density at the same mean energy
    m, st = orc.state(W.BE, *orc.moments72(W.BE, f))
    assert st == R.RLBM_W_CLAMPED_FUGACITY
    sim = R.Simulation([W.DomainSpec(nx, ny, tau, W.BE, (P, P, V, V), (tw,) * 4, accel=accel, n_wall=nw)],
                       edf=W.BE, storage=R.RLBM_F64)
    sim.init(0, W.random_domain_state(nx, ny, 3, W.BE))
    sim.set_populations(0, np.broadcast_to(f[:, None, None], (72, ny + 2, nx + 2)))
    sim.set_grid(grid)
    sim.step(1)
    g = sim.get_populations(0)
    assert sim.sync_status() & R.RLBM_W_CLAMPED_FUGACITY
    sim.close()
    zw, _ = orc.z_from_n_theta(W.BE, nw, tw)
    own = orc.feq_order(W.BE, 5, m[1], m[2] + accel[0] * tau, m[3] + accel[1] * tau, m[4], m[0], m[5])
    want = orc.feq_order(W.BE, 5, tw, 0.0, 0.0, zw) - own
    for row, cell in ((0, 1), (ny + 1, ny)):
        err = g[:, row, 1:-1] - (want[:, None] + g[:, cell, 1:-1])
        assert np.max(np.abs(err)) <= 1e-8, (row, np.max(np.abs(err)))
