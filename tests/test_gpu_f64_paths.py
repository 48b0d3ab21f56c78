"""FP64 form: the fast solvers (FP32 start, FP64 corrections; series in t = g_1) and
the general ones they hand over to, at the edges of the fast range.

An equilibrium state set with rlbm_init comes back from rlbm_moments (unstreamed)
with the fields it was set from, whichever solver runs: the fifth-order projection
keeps N^mu and T^{mu nu}. Tolerance: 2^-53 times the 72-term moment sums' growth
(about 10), the Landau and fugacity conditioning (about 10 for |u| <= 0.6 and the
fugacities below) and a factor 10 in hand: 1e-13 * 10 = 1e-12 relative."""
import numpy as np
import pytest

from paper_1709_09073_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1709_09073_gb300 import build, rlbm
    build.build()
    rlbm.load()
    return rlbm


def _round_trip(R, edf, z, theta, ux, uy):
    nx = z.size
    sim = R.Simulation([W.DomainSpec(nx, 1, 0.9, edf)], edf=edf, storage=R.RLBM_F64)
    st = sim.init(0, W.InitialState(W.INIT_Z_THETA, *[a.reshape(1, nx) for a in (z, theta, ux, uy)]))
    n, th, vx, vy, zz = [a.ravel() for a in sim.moments(0, streamed=False)]
    st |= sim.sync_status()
    sim.close()
    return st, n, th, vx, vy, zz


# fugacities across the fast range's edges (FD t = 0.2, 0.45, 0.75, 1.35 are z = 0.22,
# 0.57, 1.12, 2.86; BE z = 0.18, 0.36, 0.53, 0.74) and well outside it
@pytest.mark.parametrize("edf,zs", [
    (W.MJ, [1e-12, 1e-3, 1.0, 50.0]),
    (W.FD, [1e-9, 1e-3, 0.2, 0.2214, 0.23, 0.568, 0.569, 0.9, 1.117, 1.12, 2.85, 2.86, 2.87, 6.0, 25.0]),
    (W.BE, [1e-9, 1e-3, 0.18, 0.1813, 0.19, 0.362, 0.363, 0.527, 0.53, 0.74, 0.7408, 0.75, 0.9]),
])
def test_equilibrium_round_trip_over_fugacity(R, edf, zs):
    z = np.array(zs)
    theta = np.linspace(0.5, 2.0, z.size)
    ux, uy = np.linspace(-0.4, 0.5, z.size), np.linspace(0.3, -0.2, z.size)
    st, _, th, vx, vy, zz = _round_trip(R, edf, z, theta, ux, uy)
    assert st == 0
    assert np.max(np.abs(zz / z - 1)) <= TOL and np.max(np.abs(th / theta - 1)) <= TOL
    assert max(np.max(np.abs(vx - ux)), np.max(np.abs(vy - uy))) <= TOL


# densities across the FP32 range of the Landau start (E between 1e-15 and 1e15) and
# outside it; a power of two scales every population exactly, so u and theta keep
@pytest.mark.parametrize("exp2", [-70, -52, -49, 0, 40, 48, 52, 90])
def test_landau_scale(R, exp2):
    z = np.full(9, 0.3 * 2.0 ** exp2)
    theta = np.linspace(0.7, 1.4, 9)
    ux, uy = np.linspace(-0.5, 0.5, 9), np.linspace(0.3, 0.1, 9)
    st, _, th, vx, vy, zz = _round_trip(R, W.MJ, z, theta, ux, uy)
    assert st == 0
    assert np.max(np.abs(zz / z - 1)) <= TOL and np.max(np.abs(th / theta - 1)) <= TOL
    assert max(np.max(np.abs(vx - ux)), np.max(np.abs(vy - uy))) <= TOL
