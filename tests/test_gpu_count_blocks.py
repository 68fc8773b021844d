"""The unit-count tile pass on more tiles than its wide blocks run at once (they
take grids of few tiles), ragged and at any address, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from tests.gpu_util import u32
from tests.test_gpu_count_tiles import _fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile,shape", [(32, (641, 1027)), (32, (1, 40001)), (32, (2050, 1300)), (64, (2050, 1300)),
                                        (64, (70, 20001)), (64, (4097, 641))])
def test_count_blocks(d8, tile, shape):
    H, W = shape
    d8.set_tile(tile)
    try:
        for name, d in _fields(H, W):
            ref = oracle.accumulate(d)
            for off, pad in ((0, -W % 16), (1, 2)):
                db = torch.full((H, off + W + pad), 250, dtype=torch.uint8, device="cuda")
                db[:, off:off + W] = torch.from_numpy(d).cuda()
                A = d8.accumulate(db[:, off:off + W])
                assert d8.get_status() == "OK"
                np.testing.assert_array_equal(u32(A), ref, err_msg=f"{name} {off}")
    finally:
        d8.set_tile(64)
