"""The adjoint's combine where a block appends to the list of open exits more than
once in a launch: more exits than all blocks of a launch take in one pass, and
more than the last blocks take; path lengths (cotangent 1, exact in fp32).  And the
time of a field whose paths wind, against that of one whose paths do not."""
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
def test_last_blocks(d8, tile):
    H, W = (1001, 777) if tile == 64 else (500, 400)  # below the slot limit of the last blocks
    f = demgen.serpentine_dirs(H, W)
    d8.set_tile(tile)
    try:
        for _ in range(5):
            g = d8.accumulate_backward(to_dev(f), torch.ones((H, W), device="cuda"))
            assert d8.get_status() == "OK"
            np.testing.assert_array_equal(g.cpu().numpy(), oracle.transposed(f, np.ones((H, W))).astype(np.float32))
    finally:
        d8.set_tile(64)


@pytest.mark.parametrize("tile, n", [(32, 700), (64, 1024)])
def test_time_of_a_winding_field(d8, tile, n):
    """Below the slot limit, a boustrophedon's adjoint takes 1.6 times as long as a
    fractal's (2.9 to 3.1 times when one block went through its lists)."""
    fields = [to_dev(oracle.flowdir(demgen.fractal(n, n, seed=3, cache=False))), to_dev(demgen.serpentine_dirs(n, n))]
    w, g = torch.rand((n, n), device="cuda"), torch.empty((n, n), device="cuda")
    best = [float("inf")] * 2
    d8.set_tile(tile)
    try:
        for _ in range(20):
            for k, d in enumerate(fields):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                d8.accumulate_backward(d, w, out=g)
                a.record()
                for _ in range(10):
                    d8.accumulate_backward(d, w, out=g)
                b.record()
                b.synchronize()
                best[k] = min(best[k], a.elapsed_time(b))
        assert best[1] < 2.2 * best[0], best
    finally:
        d8.set_tile(64)
