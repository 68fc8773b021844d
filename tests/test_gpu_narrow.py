"""Unit counts of grids narrower or lower than a tile, on both sides of the line
below which they take kernels of their own, rows of codes and counts at any
address, with inflow across the first and last row; counts against the oracle,
and the time of a grid of three columns against that of a square one."""
import numpy as np
import pytest
import torch

import demgen
import oracle
from tests.gpu_util import u32
from tests.test_gpu_count_tiles import _fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile", [32, 64, 128])
@pytest.mark.parametrize("side", [1, 2, 3, 5, 8, 9, 16, 17, 32, 33])
def test_narrow_grids(d8, tile, side):
    n = 40000 // side if tile == 32 else 80000 // side  # more tiles than run at once in wide blocks
    d8.set_tile(tile)
    try:
        for H, W in ((side, n), (n, side)):
            for name, d in _fields(H, W):
                if name not in ("fractal", "spiral", "ends", "serpentine", "all 2", "all 5"):
                    continue
                ref = oracle.accumulate(d)
                for off, aoff, pad in ((0, 0, -W % 16), (3, 1, 2)):
                    db = torch.full((H, off + W + pad), 250, dtype=torch.uint8, device="cuda")
                    db[:, off:off + W] = torch.from_numpy(d).cuda()
                    Ab = torch.full((H, aoff + W + pad), 7, dtype=torch.int32, device="cuda").view(torch.uint32)
                    A = d8.accumulate(db[:, off:off + W], out=Ab[:, aoff:aoff + W])
                    assert d8.get_status() == "OK"
                    np.testing.assert_array_equal(u32(A), ref, err_msg=f"{name} {H} {W} {off}")
                    rest = Ab.view(torch.int32)
                    assert bool((rest[:, :aoff] == 7).all()) and bool((rest[:, aoff + W:] == 7).all())
                # inflow into the first row, as weights there
                top = np.random.default_rng(side).integers(0, 50, size=W).astype(np.uint32)
                w = np.ones((H, W))
                w[0] += top
                got = d8.accumulate_inflow(torch.from_numpy(d).cuda(), torch.from_numpy(top.view(np.int32)).cuda().view(torch.uint32), None)
                np.testing.assert_array_equal(u32(got), oracle.accumulate_weighted(d, w).astype(np.uint32), err_msg=name)
            bad = np.full((H, W), 2, np.uint8)
            bad[H // 2, W // 2] = 10
            d8.accumulate(torch.from_numpy(bad).cuda())
            assert d8.get_status() == "ERR_ARG"
    finally:
        d8.set_tile(64)


@pytest.mark.parametrize("tile, bound", [(64, 4.3), (32, 4.25)])
def test_time_of_three_columns(d8, tile, bound):
    """1000000 x 3 against 1732 x 1732, as many cells: 3.4 and 3.75 times as long (5.3
    and 4.75 by the kernels for full tiles)."""
    fields = [torch.from_numpy(oracle.flowdir(demgen.fractal(1732, 1732, seed=3, cache=False))).cuda(),
              torch.full((1000000, 3), 2, dtype=torch.uint8, device="cuda")]
    As = [torch.empty(d.shape, dtype=torch.uint32, device="cuda") for d in fields]
    best = [float("inf")] * 2
    d8.set_tile(tile)
    try:
        for _ in range(20):
            for k, d in enumerate(fields):
                a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
                d8.accumulate(d, out=As[k])
                a.record()
                for _ in range(10):
                    d8.accumulate(d, out=As[k])
                b.record()
                b.synchronize()
                best[k] = min(best[k], a.elapsed_time(b))
        assert best[1] < bound * best[0], best
    finally:
        d8.set_tile(64)
