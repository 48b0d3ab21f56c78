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


# nx, ny, number of domains, blocks with whole packed tiles, with one warp each; single where
# those fit in one wave: 608 blocks, 760 for FP32 without halo work and w <= 6
@pytest.mark.parametrize("storage", [F32, F32DEV, BF16, F16])
@pytest.mark.parametrize("wall", [False, True])
@pytest.mark.parametrize("nx,ny,k,whole,single", [
    (16, 1216, 1, 152, 608), (16, 1218, 1, 153, 609), (16, 4096, 1, 512, 2048), (48, 1024, 1, 384, 768),
    (33, 2000, 1, 516, 563), (1, 19456, 1, 152, 608), (1, 19457, 1, 153, 609), (1, 24320, 1, 190, 760),
    (1, 24321, 1, 191, 761), (8, 10, 202, 202, 606), (8, 10, 203, 203, 609), (6, 5, 608, 608, 608),
    (6, 5, 760, 760, 760), (6, 6, 305, 305, 610), (7, 5, 609, 609, 1218), (32, 2432, 1, 608, 608),
    (33, 2200, 1, 568, 619), (33, 2700, 1, 697, 760), (33, 2701, 1, 698, 761)])
def test_one_wave_limit(R, storage, wall, nx, ny, k, whole, single):
    bc = (W.PERIODIC, W.PERIODIC) + ((W.FIXED_T_WALL,) * 2 if wall else (W.PERIODIC,) * 2)
    specs = [W.DomainSpec(nx, ny, 0.9, W.MJ, bc)] * k
    tiles = R.rlbm_layout_tiles(specs, W.MJ, storage, True)
    assert all(c.min() == 1 and c.max() == 1 for c in coverage(specs, tiles))
    fits = single <= (760 if storage in (F32, F32DEV) and not wall and nx % 32 <= 6 else 608)
    assert len(tiles) == (single if fits else whole)
    assert np.any(tiles[:, 3] > ONE_WARP) == (fits and nx % 32 > 0)
