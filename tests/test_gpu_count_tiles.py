"""The unit-count tile pass where it can go wrong: whole and ragged tiles, at
the grid's edge and away from it, rows of any alignment, fields with one long
path, with every cell a source, with all cells meeting in one, path ends
inside and targets off the grid, and codes that are not directions; counts
against the oracle."""
import numpy as np
import pytest
import torch

import demgen
import oracle
from tests.gpu_util import DI, DJ, spiral_dirs, u32

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (2, 97), (32, 32), (64, 64), (65, 63), (128, 192), (193, 257), (320, 300)]


def _toward(H, W, ci, cj):
    """Every cell steps towards (ci, cj), diagonally first."""
    di = np.sign(ci - np.arange(H))[:, None] + np.zeros((1, W), int)
    dj = np.sign(cj - np.arange(W))[None, :] + np.zeros((H, 1), int)
    d = np.full((H, W), 9, np.uint8)
    for k in range(8):
        d[(di == DI[k]) & (dj == DJ[k])] = k
    return d


def _fields(H, W):
    rng = np.random.default_rng(H * 1000 + W)
    yield "fractal", oracle.flowdir(demgen.fractal(H, W, seed=H + W, cache=False))
    yield "spiral", spiral_dirs(H, W)
    yield "meet", _toward(H, W, H // 2, W // 3)
    for k in range(8):  # parallel paths off the grid
        yield f"all {k}", np.full((H, W), k, np.uint8)
    d = rng.integers(0, 4, size=(H, W), dtype=np.uint8)  # N, NE, E, SE: no way back west ...
    d[d == 0] = 2  # ... nor north: no cycle
    d[rng.random((H, W)) < 0.05] = 9
    d[rng.random((H, W)) < 0.05] = 8
    yield "ends", d
    if H > 1 and W > 1:
        yield "serpentine", demgen.serpentine_dirs(H, W)


@pytest.mark.parametrize("tile", [32, 64, 128])
@pytest.mark.parametrize("shape", SHAPES)
def test_count_tiles(d8, tile, shape):
    H, W = shape
    d8.set_tile(tile)
    try:
        for name, d in _fields(H, W):
            ref = oracle.accumulate(d)
            for off, pad, aoff in ((0, -W % 16, 0), (1, 2, 1)):
                db = torch.full((H, off + W + pad), 250, dtype=torch.uint8, device="cuda")
                db[:, off:off + W] = torch.from_numpy(d).cuda()
                Ab = torch.full((H, aoff + W + -W % 4), 7, dtype=torch.int32, device="cuda").view(torch.uint32)
                A = d8.accumulate(db[:, off:off + W], out=Ab[:, aoff:aoff + W])
                assert d8.get_status() == "OK"
                np.testing.assert_array_equal(u32(A), ref, err_msg=f"{name} {off}")
                rest = Ab.view(torch.int32)
                assert bool((rest[:, :aoff] == 7).all()) and bool((rest[:, aoff + W:] == 7).all())
            if H * W > 1:  # a code that is none: reported, and its path ends there
                bad = d.copy()
                bad[H // 2, W // 2] = 10
                d8.accumulate(torch.from_numpy(bad).cuda())
                assert d8.get_status() == "ERR_ARG"
    finally:
        d8.set_tile(64)
