"""The fill's tile passes where they can go wrong: sides around the tile size
and the warp size, paths that wind through a tile many times, elevations of
both signs and zero, no epsilon, and rows that are not aligned; bit for bit
against the oracle's priority flood."""
import numpy as np
import pytest
import torch

import demgen
import oracle

pytestmark = pytest.mark.gpu

SHAPES = [(3, 700), (63, 65), (64, 64), (66, 127), (97, 33), (129, 191), (193, 256), (320, 66), (577, 643)]  # the last with coarse levels


def _surfaces(H, W):
    rng = np.random.default_rng(H * 1000 + W)
    yield "fractal", demgen.fractal_raw(H, W, seed=H * 7 + W) - np.float32(500.0)
    yield "pits", rng.integers(-3, 4, size=(H, W)).astype(np.float32) * np.float32(0.5)
    z = np.ascontiguousarray(demgen.serpentine_dem(577, 700)[:H, :W])
    z[H // 2, W // 2] = z.max()  # a dam across the channel: everything above it fills
    yield "serpentine", z


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("eps", [0.0, 1e-3])
def test_fill_tiles(d8, shape, eps):
    H, W = shape
    for name, z in _surfaces(H, W):
        ref = oracle.fill_eps(z, eps)
        buf = torch.full((H, W + 3), -7.0, device="cuda")
        buf[:, 1:W + 1] = torch.from_numpy(z).cuda()
        out = torch.full((H, W + 5), -9.0, device="cuda")
        d8.fill(buf[:, 1:W + 1], eps, out=out[:, 3:W + 3])
        assert d8.get_status() == "OK"
        np.testing.assert_array_equal(out[:, 3:W + 3].cpu().numpy(), ref, err_msg=name)
        assert bool((out[:, :3] == -9.0).all()) and bool((out[:, W + 3:] == -9.0).all())
