"""The top level's walks where they are long: chains through thousands of units'
exits, with and without other paths joining them; counts and areas of
whole-number weights (sums below 2^24, so exact) against the oracle."""
import numpy as np
import pytest
import torch

import demgen
import oracle
from tests.gpu_util import spiral_dirs, to_dev, u32

pytestmark = pytest.mark.gpu


def _joined(H, W):
    """A boustrophedon in which a cell of every fourth row, every 37 columns,
    goes straight on to the next row: a short cut, and the rest a branch."""
    d = demgen.serpentine_dirs(H, W)
    cut = np.zeros((H, W), bool)
    cut[2:H - 1:4, 5::37] = True
    d[cut & (d != 9)] = 4
    return d


@pytest.mark.parametrize("tile", [32, 64, 128])
@pytest.mark.parametrize("shape", [(1100, 1030), (70, 4100), (2100, 600)])
def test_long_top_walks(d8, tile, shape):
    H, W = shape
    fields = {"serpentine": demgen.serpentine_dirs(H, W), "spiral": spiral_dirs(H, W), "joined": _joined(H, W)}
    w = np.random.default_rng(H + W).integers(0, 8, size=shape).astype(np.float32)
    assert w.sum() < 2 ** 24
    d8.set_tile(tile)
    try:
        for name, d in fields.items():
            dt = to_dev(d)
            np.testing.assert_array_equal(u32(d8.accumulate(dt)), oracle.accumulate(d), err_msg=name)
            A = d8.accumulate_weighted(dt, torch.from_numpy(w).cuda()).cpu().numpy()
            np.testing.assert_array_equal(A, oracle.accumulate_weighted(d, w.astype(np.float64)), err_msg=name)
            assert d8.get_status() == "OK"
    finally:
        d8.set_tile(64)
