"""The mixed storages' read-out writes its FP32 and double-float values as FP64 on the
integer pipe. theta and z are FP32 values: every FP64 output has 29 zero low bits. n, u
of a rest state with a power-of-two density (the binade edge, where the ulp halves)
and of states at u = 0, tiny u and either sign agree with the FP64 read-out of the same
populations in FP64 storage to FP32 rounding (1e-6 of n and theta, 1e-6 absolute in u)."""
import numpy as np
import pytest

from paper_1709_09073_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["RLBM_F32", "RLBM_F32DEV"])
@pytest.mark.parametrize("u0", [0.0, 1e-12, 1e-3, -0.3])
def test_readout_matches_fp64(storage, u0):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1709_09073_gb300 import build, rlbm as R
    build.build()
    R.load()
    ny, nx = 7, 41
    rng = np.random.default_rng(5)
    n = np.where(rng.uniform(size=(ny, nx)) < 0.5, 2.0, 1.0 + 1e-3 * rng.standard_normal((ny, nx)))
    th = 1.0 + 0.05 * rng.standard_normal((ny, nx))
    ux, uy = u0 * np.ones((ny, nx)), u0 * rng.uniform(-1, 1, (ny, nx))
    out = []
    for st in (getattr(R, storage), R.RLBM_F64):
        sim = R.Simulation([W.DomainSpec(nx, ny, 0.9)], edf=W.MJ, storage=st)
        assert sim.init(0, W.InitialState(W.INIT_N_THETA, n, th, ux, uy)) == 0
        out.append(sim.moments(0, streamed=False))
        sim.close()
    a, b = out
    for k in (1, 4):
        assert not (a[k].view(np.uint64) & np.uint64((1 << 29) - 1)).any()
    assert np.max(np.abs(a[0] / b[0] - 1)) <= 1e-6 and np.max(np.abs(a[1] / b[1] - 1)) <= 1e-6
    assert max(np.max(np.abs(a[k] - b[k])) for k in (2, 3)) <= 1e-6
