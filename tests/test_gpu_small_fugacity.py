"""FP64 form, FD and BE at small fugacities: the Newton residuals of the series solve are
of order one whatever the fugacity, so a dilute gas is solved as well as a dense one.

An equilibrium state set from (z, theta, u) reads back (unstreamed) as what it was set
from; temperatures and tolerance (1e-12) are those of the round trip over the other
fugacities (test_gpu_f64_paths.py)."""
import numpy as np
import pytest

from paper_1709_09073_gb300 import workloads as W

pytestmark = pytest.mark.gpu
TOL = 1e-12


@pytest.mark.parametrize("edf", [W.FD, W.BE])
@pytest.mark.parametrize("z", [1e-25, 9e-21, 1e-20, 1e-19, 1e-18, 1e-17, 1e-16, 3e-16, 1e-15, 1e-14, 1e-12, 1e-10])
def test_round_trip(edf, z):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1709_09073_gb300 import build, rlbm as R
    build.build()
    R.load()
    nx = 64
    th = np.linspace(0.5, 2.0, nx).reshape(1, nx)
    zz = z * np.linspace(0.9, 1.1, nx).reshape(1, nx)
    ux, uy = np.linspace(-0.4, 0.4, nx).reshape(1, nx), np.full((1, nx), 0.2)
    sim = R.Simulation([W.DomainSpec(nx, 1, 0.9, edf)], edf=edf, storage=R.RLBM_F64)
    st = sim.init(0, W.InitialState(W.INIT_Z_THETA, zz, th, ux, uy))
    n, t, vx, vy, z2 = sim.moments(0, streamed=False)
    st |= sim.sync_status()
    sim.close()
    assert st == 0
    assert np.max(np.abs(z2 / zz - 1)) <= TOL and np.max(np.abs(t / th - 1)) <= TOL
    # dilute: g_2 = z to z / 4
    assert np.max(np.abs(n / (2 * np.pi * th * th * zz) - 1)) <= TOL + z
    assert max(np.max(np.abs(vx - ux)), np.max(np.abs(vy - uy))) <= TOL
