"""16-bit storages: the FD/BE fugacity by series in t = g_1 (collision: w up to 0.48;
initialiser and wall ghosts: G = g_2 up to 0.25) and the Newton solve beyond, at the
edges of both.

Each domain is at rest in its own reference state (deviations zero up to FP32
rounding), so rounding to 16 bits plays no part: the fields read back, before and
after steps, are the state itself. Tolerance: FP32 rounding of n and eps (2^-23, the
sum of a few) times the conditioning of z, d ln z / d ln R up to about 10 for the BE
states below, times 4 in hand: 1.2e-7 * 2 * 10 * 4 = 1e-5."""
import numpy as np
import pytest

from paper_1709_09073_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-5


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1709_09073_gb300 import build, rlbm
    build.build()
    rlbm.load()
    return rlbm


def _g2(z, edf):
    k = np.arange(1, 4000)
    if edf == W.BE:
        return float(np.sum(z ** k / k ** 2.0))
    x, w = np.polynomial.legendre.leggauss(400)
    x = 30.0 * (x + 1)
    return float(np.sum(30.0 * w * x / (np.exp(x) / z + 1)))


# FD w = 0.48 is z = 0.62, G = 0.25 is z = 0.267; BE z = 0.38 and 0.236
@pytest.mark.parametrize("storage", ["RLBM_BF16DEV", "RLBM_F16DEV"])
@pytest.mark.parametrize("edf,zs", [(W.FD, [1e-3, 0.1, 0.26, 0.27, 0.3, 0.6, 0.61, 0.62, 0.63, 0.7, 2.0, 6.0]),
                                    (W.BE, [1e-3, 0.1, 0.23, 0.24, 0.3, 0.375, 0.38, 0.385, 0.4, 0.6])])
def test_rest_states_over_fugacity(R, storage, edf, zs):
    doms, theta = [], np.linspace(0.8, 1.25, len(zs))
    for z, th in zip(zs, theta):
        n = 2 * np.pi * th * th * _g2(z, edf)
        doms.append(W.DomainSpec(5, 3, 0.8, edf, ref_n=n, ref_theta=float(th)))
    sim = R.Simulation(doms, edf=edf, storage=getattr(R, storage))
    one = np.ones((3, 5))
    st = 0
    for i, (d, th) in enumerate(zip(doms, theta)):
        st |= sim.init(i, W.InitialState(W.INIT_N_THETA, d.ref_n * one, th * one, 0 * one, 0 * one))
    for steps in (0, 3):
        sim.step(steps)
        for i, (d, z, th) in enumerate(zip(doms, zs, theta)):
            n, t, ux, uy, zz = sim.moments(i)
            assert np.max(np.abs(n / d.ref_n - 1)) <= TOL and np.max(np.abs(t / th - 1)) <= TOL, (z, steps)
            assert np.max(np.abs(zz / z - 1)) <= TOL and max(np.max(np.abs(ux)), np.max(np.abs(uy))) <= TOL, (z, steps)
    st |= sim.sync_status()
    sim.close()
    assert st == 0
