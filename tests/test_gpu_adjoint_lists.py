"""The adjoint's combine where a block appends to the list of open exits more than
once in a launch: more exits than all blocks of a launch take in one pass, and
more than the last block takes; path lengths (cotangent 1, exact in fp32)."""
import numpy as np
import pytest
import torch

import demgen
import oracle
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


def test_launched_rounds(d8):
    n = 8192  # parallel paths east: 127 exits in each row, a million in all
    g = d8.accumulate_backward(torch.full((n, n), 2, dtype=torch.uint8, device="cuda"), torch.ones((n, n), device="cuda"))
    assert d8.get_status() == "OK"
    assert torch.equal(g, torch.arange(n, 0, -1, dtype=torch.float32, device="cuda").expand(n, n))


@pytest.mark.parametrize("tile", [32, 64])
def test_last_block(d8, tile):
    H, W = (1001, 777) if tile == 64 else (500, 400)  # below the slot limit of the last block
    f = demgen.serpentine_dirs(H, W)
    d8.set_tile(tile)
    try:
        for _ in range(5):
            g = d8.accumulate_backward(to_dev(f), torch.ones((H, W), device="cuda"))
            assert d8.get_status() == "OK"
            np.testing.assert_array_equal(g.cpu().numpy(), oracle.transposed(f, np.ones((H, W))).astype(np.float32))
    finally:
        d8.set_tile(64)
