"""The direction stencil's inside and edge loops against the oracle: sides
around whole tiles (so that some items lie inside the grid and some on its
edge), rows of every alignment of z and of the codes, ties, exact zeros,
non-finite elevations inside and at the edge, every rule and tile side."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1), (3, 5), (64, 64), (65, 131), (130, 66), (193, 260), (258, 391)]


def _surfaces(H, W):
    rng = np.random.default_rng(H * 1000 + W)
    yield "smooth", (np.add.outer(np.arange(H), 0.7 * np.arange(W)) + rng.random((H, W)) * 3.0).astype(np.float32)
    yield "ties", rng.integers(-2, 3, size=(H, W)).astype(np.float32)  # flats, equal drops, zeros
    yield "tiny", (rng.standard_normal((H, W)) * 1e-40).astype(np.float32)  # subnormal differences
    z = (rng.standard_normal((H, W)) * 100.0).astype(np.float32)
    bad = rng.random((H, W)) < 0.002
    bad[H // 2, W // 2] = True
    z[bad] = rng.choice(np.array([np.nan, np.inf, -np.inf], dtype=np.float32), size=int(bad.sum()))
    yield "nonfinite", z


@pytest.mark.parametrize("tile", [32, 64, 128])
@pytest.mark.parametrize("rule", ["steepest", "lowest", "steepest_nodata", "lowest_nodata"])
@pytest.mark.parametrize("shape", SHAPES)
def test_flowdir_rows(d8, tile, rule, shape):
    H, W = shape
    d8.set_tile(tile)
    try:
        for name, z in _surfaces(H, W):
            ref = oracle.flowdir(z, rule, allow_nonfinite=True)
            for zoff, zpad, doff, dpad in ((0, -W % 4, 0, -W % 4), (1, 2, 0, -W % 4), (0, -W % 4, 3, 2), (2, 7, 1, 0)):
                zb = torch.full((H, zoff + W + zpad), -5e4, device="cuda")
                zb[:, zoff:zoff + W] = torch.from_numpy(z).cuda()
                db = torch.full((H, doff + W + dpad), 77, dtype=torch.uint8, device="cuda")
                d8.flowdir(zb[:, zoff:zoff + W], rule, out=db[:, doff:doff + W])
                want = "ERR_NONFINITE" if name == "nonfinite" and "nodata" not in rule else "OK"
                assert d8.get_status() == want
                np.testing.assert_array_equal(db[:, doff:doff + W].cpu().numpy(), ref, err_msg=f"{name} {zoff} {zpad} {doff}")
                assert bool((db[:, :doff] == 77).all()) and bool((db[:, doff + W:] == 77).all())
    finally:
        d8.set_tile(64)
