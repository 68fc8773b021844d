"""The weighted finalise where it can go wrong: whole and ragged tiles of each
side, rows of codes at any address, fields whose receivers' paths are one long
chain, meet in one cell or end inside.  Weights are whole numbers whose sums
stay below 2^24, so every rounding is exact and areas equal the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from tests.test_gpu_count_tiles import _fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [32, 64, 128])
@pytest.mark.parametrize("shape", [(1, 300), (65, 63), (128, 192), (193, 257), (320, 300), (70, 1100)])
def test_area_finalise(d8, tile, shape):
    H, W = shape
    w = np.random.default_rng(7 * H + W).integers(0, 128, size=shape).astype(np.float32)
    assert w.sum() < 2 ** 24
    d8.set_tile(tile)
    try:
        for name, d in _fields(H, W):
            ref = oracle.accumulate_weighted(d, w.astype(np.float64))
            for off, pad in ((0, -W % 16), (1, 2), (2, 1), (3, 0)):
                db = torch.full((H, off + W + pad), 250, dtype=torch.uint8, device="cuda")
                db[:, off:off + W] = torch.from_numpy(d).cuda()
                A = d8.accumulate_weighted(db[:, off:off + W], torch.from_numpy(w).cuda()).cpu().numpy()
                assert d8.get_status() == "OK"
                np.testing.assert_array_equal(A, ref, err_msg=f"{name} {off}")
    finally:
        d8.set_tile(64)
