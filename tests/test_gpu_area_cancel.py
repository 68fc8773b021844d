"""Weighted areas whose inflow into a tile cancels but for its low part: two paths
meet in one cell of another tile, one with 1000 + t, the other with -1000, where
1000 + t needs more than an fp32's bits.  Every sum is a multiple of 2^-30 that a
float-float number holds exactly, so areas equal the oracle's.  The cell lies
beyond the border of a tile, of a group of each level and of a top-level unit,
one path or both coming across it."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("strategy", ["ring", "jump"])
@pytest.mark.parametrize("tile", [32, 64, 128])
def test_cancelling_inflow(d8, tile, strategy):
    d8.set_tile(tile)
    d8.set_strategy(strategy)
    try:
        for i, j in ((1, tile), (tile, tile), (tile, 256), (256, tile), (1, 512), (512, 512)):  # the cell where they meet
            H, W = i + 3, j + 70
            # beside the border from the west; the other from the north-west (both across it) or the north
            beside = [(i, j - 2, 2), (i, j - 1, 2)]
            both = [(i - 1, j - 2, 2), (i - 1, j - 1, 3)]
            north = [(i - 1, j + 2, 6), (i - 1, j + 1, 6), (i - 1, j, 4)]
            for other in (both, north) if i > 1 else (both,):  # (row 0 is in row 1's tile)
                d = np.full((H, W), 8, np.uint8)
                d[i, j:W - 1] = 2
                for a, b, k in beside + other:
                    d[a, b] = k
                for first, second in ((beside, other), (other, beside)):
                    for big, t in ((1000.0, 2.0 ** -30), (-1000.0, 2.0 ** -30), (1000.0, -77 * 2.0 ** -30), (1.0, 2.0 ** -60)):
                        w = np.zeros((H, W), np.float32)
                        w[first[0][:2]] = big
                        w[first[1][:2]] = t
                        w[second[0][:2]] = -big
                        ref = np.zeros((H, W))  # (1000 + t has more bits than the oracle's fp64 when t is 2^-60)
                        for path in (first, second):
                            s = 0.0
                            for a, b, _ in path:
                                s += float(w[a, b])
                                ref[a, b] = s
                        ref[i, j:] = t
                        if abs(t) > 2.0 ** -40:
                            np.testing.assert_array_equal(oracle.accumulate_weighted(d, w.astype(np.float64)), ref)
                        A = d8.accumulate_weighted(torch.from_numpy(d).cuda(), torch.from_numpy(w).cuda()).cpu().numpy()
                        assert d8.get_status() == "OK"
                        np.testing.assert_array_equal(A, ref.astype(np.float32), err_msg=f"{i} {j} {big} {t}")
    finally:
        d8.set_tile(64)
        d8.set_strategy("ring")
