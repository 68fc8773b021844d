"""The single-launch combine and the finalise from the receivers' inflow at the
sides where the route changes (one tile, one group, one more than a group),
for single calls, batches and strips; counts against the oracle."""
import numpy as np
import pytest
import torch

import demgen
import oracle
from paper_1605_05773_gb300 import strips
from tests.gpu_util import spiral_dirs, to_dev, u32

pytestmark = pytest.mark.gpu


def _shapes(tile):
    g = 512 if tile == 128 else 8 * tile
    return [(tile, tile), (tile + 1, 7), (g - 1, g), (g, 2 * tile - 1), (g + 1, tile), (70, g + 5)]


@pytest.mark.parametrize("tile", [32, 64, 128])
@pytest.mark.parametrize("strategy", ["ring", "lane_mask", "jump"])
def test_small_grids(d8, tile, strategy):
    d8.set_tile(tile)
    d8.set_strategy(strategy)
    try:
        for H, W in _shapes(tile):
            z = demgen.fractal(H, W, seed=H + W, cache=False)
            d, A = d8.flowdir_accumulate(to_dev(z))
            assert d8.get_status() == "OK"
            ref = oracle.flowdir(z)
            np.testing.assert_array_equal(d.cpu().numpy(), ref)
            np.testing.assert_array_equal(u32(A), oracle.accumulate(ref))
            s = spiral_dirs(H, W)
            np.testing.assert_array_equal(u32(d8.accumulate(to_dev(s))), oracle.accumulate(s))
            assert d8.get_status() == "OK"
    finally:
        d8.set_tile(64)
        d8.set_strategy("ring")


@pytest.mark.parametrize("tile", [32, 64])
def test_small_batches(d8, tile):
    d8.set_tile(tile)
    try:
        for shapes in ([(5, 9), (tile, tile)], _shapes(tile)[:4], _shapes(tile)):
            zs = [demgen.fractal(h, w, seed=7 * h + w, cache=False) for h, w in shapes]
            plan = d8.BatchPlan(shapes)
            for _ in range(2):
                dirs, As = plan.run([to_dev(z) for z in zs])
                assert d8.get_status() == "OK"
                for z, d, A in zip(zs, dirs, As):
                    np.testing.assert_array_equal(d.cpu().numpy(), oracle.flowdir(z))
                    np.testing.assert_array_equal(u32(A), oracle.accumulate(oracle.flowdir(z)))
            plan.close()
    finally:
        d8.set_tile(64)


@pytest.mark.parametrize("shape,n", [((90, 60), 3), ((300, 257), 4), ((1200, 500), 2)])
def test_strips_of_small_grids(d8, shape, n):
    z = demgen.fractal(*shape, seed=11, cache=False)
    d, A = strips.flowdir_accumulate_strips(z, n)
    np.testing.assert_array_equal(np.asarray(d), oracle.flowdir(z))
    np.testing.assert_array_equal(np.asarray(A).view(np.uint32), oracle.accumulate(oracle.flowdir(z)))
