"""rlbm_layout_tiles(packed = 1) reports what a handle walks (host logic): small mixed
launches list their packed tiles one warp at a time (w + 256), and every cell is covered
exactly once under the kernels' lane mapping, restated here."""
import numpy as np
import pytest

from paper_1709_09073_gb300 import workloads as W

TILE_W, TILE_H, ONE_WARP = 32, 4, 256
F64, F32, BF16, F16, F32DEV = 0, 1, 2, 3, 4


@pytest.fixture(scope="module")
def R():
    from paper_1709_09073_gb300 import build, rlbm
    rlbm.load(build.build())
    return rlbm


def coverage(specs, tiles):
    counts = [np.zeros((s.ny, s.nx), dtype=np.int64) for s in specs]
    for d, x0, y0, w in ((int(v) for v in t) for t in tiles):
        for warp in range(TILE_H if w < ONE_WARP else 1):
            lane = np.arange(TILE_W)
            if w == 0:
                x, y = x0 + lane, np.full(TILE_W, y0 + warp)
            else:
                k = w % ONE_WARP
                r = TILE_W // k
                lane = lane[lane < r * k]
                x, y = x0 + lane % k, y0 + warp * r + lane // k
            keep = (x < specs[d].nx) & (y < specs[d].ny)
            np.add.at(counts[d], (y[keep], x[keep]), 1)
    return counts


@pytest.mark.parametrize("storage", [F64, F32, BF16, F16, F32DEV])
@pytest.mark.parametrize("edf", [W.MJ, W.FD, W.BE])
def test_small_launches(R, edf, storage):
    specs = [W.DomainSpec(nx, ny, 0.9, edf) for nx in (1, 3, 16, 17, 33, 47) for ny in (1, 7, 33)]
    tiles = R.rlbm_layout_tiles(specs, edf, storage, True)
    assert all(c.min() == 1 and c.max() == 1 for c in coverage(specs, tiles))
    packed = tiles[tiles[:, 3] > 0]
    assert len(packed) and np.all((packed[:, 3] > ONE_WARP) == (storage != F64))
    for d, x0, y0, w in packed:
        nx, k = specs[d].nx, w % ONE_WARP
        assert 1 <= k <= 16 and x0 == (nx - 1) // TILE_W * TILE_W and k == nx - x0
        assert y0 < specs[d].ny and y0 % ((TILE_H if storage == F64 else 1) * (TILE_W // k)) == 0
