"""Launches of few tiles: the FP64 step by three warps per 32 cells against the
one-thread-per-cell step (a persistent grid of one block selects it), and the mixed
step's packed tiles at one warp per block against the TMA-staged variant (plain
tiles). Both pairs do the same operations on the same operands in the same order, so
the populations, halo included, are equal bit for bit."""
import numpy as np
import pytest

from paper_1709_09073_gb300 import workloads as W

pytestmark = pytest.mark.gpu
P, Z, T, V = W.PERIODIC, W.ZERO_GRADIENT, W.FIXED_T_WALL, W.VELOCITY_WALL
FORCE = dict(accel=(2e-4, -1e-4))


@pytest.fixture(scope="module")
def R():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1709_09073_gb300 import build, rlbm
    build.build()
    rlbm.load()
    return rlbm


def _run(R, specs, edf, storage, select, hurt):
    sim = R.Simulation(specs, edf=edf, storage=storage)
    for i, d in enumerate(specs):
        sim.init(i, W.random_domain_state(d.nx, d.ny, 31 + i, edf, u_amp=0.05))
    if hurt:  # a non-physical cell: streamed, not relaxed, its ghosts written all the same
        f = sim.get_populations(0)
        f[:, 1, 1] = -1.0
        sim.set_populations(0, f)
    select(sim)
    sim.step(5)
    out = [sim.get_populations(i) for i in range(len(specs))]
    st = sim.sync_status()
    sim.close()
    return out, st


# full and ragged rows, one packed row per lane (w = 1), a single cell, more rows than
# a tile; every boundary, the local tau, the force; 72 tiles (the largest split launch)
@pytest.mark.parametrize("edf", [W.MJ, W.FD, W.BE])
@pytest.mark.parametrize("nx,ny,bc,more", [
    (64, 64, (P, P, P, P), {}), (33, 35, (Z, Z, Z, Z), dict(eta_s=0.5)), (45, 5, (T, Z, P, P), {}),
    (8, 41, (P, P, V, V), FORCE), (7, 9, (V, V, V, V), dict(eta_s=0.4, **FORCE)), (1, 1, (P, P, T, V), {}),
    (96, 96, (T, T, T, T), {})])
@pytest.mark.parametrize("hurt", [False, True])
def test_split_step_is_the_plain_step(R, edf, nx, ny, bc, more, hurt):
    specs = [W.DomainSpec(nx, ny, 0.9, edf, bc, (1.03,) * 4, **more)]
    a, sa = _run(R, specs, edf, R.RLBM_F64, lambda s: None, hurt)
    b, sb = _run(R, specs, edf, R.RLBM_F64, lambda s: s.set_grid(1), hurt)
    assert sa == sb
    assert all(np.array_equal(x, y, equal_nan=True) for x, y in zip(a, b))


@pytest.mark.parametrize("storage", ["RLBM_F32DEV", "RLBM_F16DEV"])
@pytest.mark.parametrize("nx,ny", [(1, 1), (33, 31), (33, 33), (65, 130), (37, 7), (48, 9), (47, 12)])
def test_one_warp_packed_tiles(R, storage, nx, ny):
    specs = [W.DomainSpec(nx, ny, 0.9, W.MJ), W.DomainSpec(nx + 2, ny + 1, 1.2, W.MJ)]
    a, sa = _run(R, specs, W.MJ, getattr(R, storage), lambda s: None, False)
    b, sb = _run(R, specs, W.MJ, getattr(R, storage), lambda s: s.select_kernel(R.RLBM_KERNEL_TMA), False)
    assert sa == sb == 0
    assert all(np.array_equal(x, y) for x, y in zip(a, b))
