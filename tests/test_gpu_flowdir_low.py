"""The direction stencil on grids lower than a tile, alone and as strips of a
taller grid; codes against the oracle, and their time against that of a square
grid of as many cells."""
import numpy as np
import pytest
import torch

import demgen
import oracle
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [32, 64, 128])
@pytest.mark.parametrize("H", [1, 2, 7, 8, 9, 31, 33, 63, 100, 127, 129])
def test_low_grids(d8, tile, H):
    W = 1500 + H
    z = demgen.fractal_raw(H + 2, W, seed=H)
    d8.set_tile(tile)
    try:
        for rule in ("steepest", "lowest_nodata"):
            got = d8.flowdir(to_dev(z[:H]), rule).cpu().numpy()
            np.testing.assert_array_equal(got, oracle.flowdir(np.ascontiguousarray(z[:H]), rule))
            got = d8.flowdir_strip(to_dev(z)[1:H + 1], 3, rule).cpu().numpy()
            np.testing.assert_array_equal(got, oracle.flowdir(z, rule)[1:H + 1])
        assert d8.get_status() == "OK"
    finally:
        d8.set_tile(64)


@pytest.mark.parametrize("tile", [32, 64, 128])
def test_time_of_a_low_grid(d8, tile):
    """8 x 400000 takes about as long as 1792 x 1792 (14 us; 23 to 33 when most of
    its work items had no rows)."""
    zs = [torch.rand(s, device="cuda") for s in ((1792, 1792), (8, 400000))]
    ds = [torch.empty(z.shape, dtype=torch.uint8, device="cuda") for z in zs]
    best = [float("inf")] * 2
    d8.set_tile(tile)
    try:
        for _ in range(30):
            for k in range(2):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                d8.flowdir(zs[k], out=ds[k])
                a.record()
                for _ in range(20):
                    d8.flowdir(zs[k], out=ds[k])
                b.record()
                b.synchronize()
                best[k] = min(best[k], a.elapsed_time(b))
        assert best[1] < 1.4 * best[0], best
    finally:
        d8.set_tile(64)
