"""The adjoint's combine where its rounds are split between launches and one
last block: fields whose paths cross far more tiles than the grid is wide, on
grids on both sides of the slot limit, and lists of every length around a
block's pass; path lengths (cotangent 1, exact in fp32) against the oracle."""
import numpy as np
import pytest
import torch

import demgen
import oracle
from tests.gpu_util import spiral_dirs, to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [32, 64])
@pytest.mark.parametrize("shape", [(64, 65), (130, 257), (333, 190), (600, 700), (1030, 1025), (2100, 600)])
def test_adjoint_rounds(d8, tile, shape):
    H, W = shape
    d8.set_tile(tile)
    try:
        for f in (demgen.serpentine_dirs(H, W), np.ascontiguousarray(demgen.serpentine_dirs(W, H).T),
                  spiral_dirs(H, W), oracle.flowdir(demgen.fractal(H, W, seed=H + W, cache=False))):
            f = np.where(f > 9, 9, f).astype(np.uint8)
            try:
                ref = oracle.transposed(f, np.ones((H, W)))
            except oracle.OracleError:  # the transposed field's codes may close loops: reported, not solved
                d8.accumulate_backward(to_dev(f), torch.ones((H, W), device="cuda"))
                assert d8.get_status() == "ERR_CYCLE"
                continue
            got = d8.accumulate_backward(to_dev(f), torch.ones((H, W), device="cuda"))
            assert d8.get_status() == "OK"
            np.testing.assert_array_equal(got.cpu().numpy().astype(np.float64), ref)
    finally:
        d8.set_tile(64)
