"""Which FP64 step a launch takes, read from a captured step's graph (kernel name, grid and
block): the step of few tiles by default up to 76 tiles, one block of the plain step per
tile beyond, and whatever the number of tiles (one included) the plain step with exactly
the grid that rlbm_set_grid asked for. At both sides of the limit the two steps give the
same populations bit for bit."""
import re

import numpy as np
import pytest

from paper_1709_09073_gb300 import workloads as W

pytestmark = [pytest.mark.gpu, pytest.mark.filterwarnings("ignore:DEBUG")]


def _step(tmp_path, nx, ny, grid, edf=W.MJ):
    """Kernel name, blocks and block shape of one captured step, and the populations after
    five launched ones."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1709_09073_gb300 import build, rlbm as R
    build.build()
    R.load()
    s = torch.cuda.Stream()
    sim = R.Simulation([W.DomainSpec(nx, ny, 0.9, edf)], edf=edf, storage=R.RLBM_F64, stream=s)
    sim.init(0, W.random_domain_state(nx, ny, 4, edf, u_amp=0.05))
    sim.set_grid(grid)
    sim.step(5)
    out = sim.get_populations(0)
    g = torch.cuda.CUDAGraph(keep_graph=True)
    with torch.cuda.graph(g, stream=s):
        sim.step(1)
    dot = tmp_path / "step.dot"
    g.debug_dump(str(dot))
    sim.close()
    name, blocks, block = re.search(r"\|\s*(\w*k_step_f64\w*)\\<\\<\\<\{?(\d+)[^,]*,\\?\{?([\d,]+)", dot.read_text()).groups()
    return "split" in name, int(blocks), block, out


@pytest.mark.parametrize("nx,ny,grid,split,blocks", [
    (1, 1, 0, True, 4), (1, 1, 1, False, 1), (7, 9, 0, True, 4), (7, 9, 1, False, 1),
    (32, 8, 0, True, 8), (32, 8, 2, False, 2), (32, 8, 5, False, 5),
    (32, 304, 0, True, 304), (32, 304, 76, False, 76), (32, 308, 0, False, 77), (32, 308, 77, False, 77)])
def test_kernel_and_grid(tmp_path, nx, ny, grid, split, blocks):
    got = _step(tmp_path, nx, ny, grid)
    assert got[:3] == (split, blocks, "32,3" if split else "32,4")


@pytest.mark.parametrize("edf", [W.MJ, W.FD, W.BE])
@pytest.mark.parametrize("nx,ny", [(1, 1), (7, 9), (32, 304), (32, 308)])
def test_same_populations(tmp_path, edf, nx, ny):
    a, b = _step(tmp_path, nx, ny, 0, edf), _step(tmp_path, nx, ny, 1, edf)
    assert not b[0] and np.array_equal(a[3], b[3])
