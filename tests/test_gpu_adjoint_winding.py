"""The adjoint on paths that wind along the columns and along the rows, on grids on
both sides of the slot limit of the combine's last launch: path lengths
(cotangent 1, exact in fp32) against the oracle.  And a cycle among the exits."""
import numpy as np
import pytest
import torch

import demgen
import oracle
from tests.gpu_util import spiral_dirs, to_dev

pytestmark = pytest.mark.gpu

_TRANSPOSED = np.arange(256, dtype=np.uint8)
_TRANSPOSED[:8] = [6, 5, 4, 3, 2, 1, 0, 7]  # codes of a field seen along its other diagonal


@pytest.mark.parametrize("tile", [32, 64])
@pytest.mark.parametrize("shape", [(64, 65), (130, 257), (333, 190), (600, 700), (1001, 777), (1030, 1025), (2100, 600)])
def test_adjoint_winding(d8, tile, shape):
    H, W = shape
    columns = _TRANSPOSED[np.ascontiguousarray(demgen.serpentine_dirs(W, H).T)]
    d8.set_tile(tile)
    try:
        for name, f in (("columns", columns), ("rows", demgen.serpentine_dirs(H, W)), ("spiral", spiral_dirs(H, W)),
                        ("spiral, transposed", _TRANSPOSED[np.ascontiguousarray(spiral_dirs(W, H).T)])):
            ref = oracle.transposed(f, np.ones((H, W)))
            assert ref.max() == H * W  # one path
            got = d8.accumulate_backward(to_dev(f), torch.ones((H, W), device="cuda"))
            assert d8.get_status() == "OK"
            np.testing.assert_array_equal(got.cpu().numpy(), ref.astype(np.float32), err_msg=name)
        rows, end = demgen.serpentine_dirs(H, W), 0 if H % 2 == 0 else W - 1
        rows[H - 1, end] = 0  # the path's end, back up into the row before
        with pytest.raises(oracle.OracleError):
            oracle.transposed(rows, np.ones((H, W)))
        d8.accumulate_backward(to_dev(rows), torch.ones((H, W), device="cuda"))
        assert d8.get_status() == "ERR_CYCLE"
    finally:
        d8.set_tile(64)
