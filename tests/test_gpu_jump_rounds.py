"""The top level by pointer jumping: few and many rounds, odd and even, on grids
of one row or column of units and of several; counts and areas of whole-number
weights (sums below 2^24, so exact) against the oracle."""
import numpy as np
import pytest
import torch

import demgen
import oracle
from tests.gpu_util import spiral_dirs, to_dev, u32

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(513, 1), (1, 1100), (1, 4200), (520, 1030), (1100, 1030)])
def test_jump_rounds(d8, shape):
    H, W = shape
    fields = {"fractal": oracle.flowdir(demgen.fractal(H, W, seed=H, cache=False)), "spiral": spiral_dirs(H, W),
              "east": np.full((H, W), 2, np.uint8)}
    if H > 1 and W > 1:
        fields["serpentine"] = demgen.serpentine_dirs(H, W)
    w = np.random.default_rng(H + W).integers(0, 8, size=shape).astype(np.float32)
    assert w.sum() < 2 ** 24
    d8.set_strategy("jump")
    try:
        for name, d in fields.items():
            dt = to_dev(d)
            for _ in range(2):  # the second call finds the workspace of the first
                np.testing.assert_array_equal(u32(d8.accumulate(dt)), oracle.accumulate(d), err_msg=name)
                A = d8.accumulate_weighted(dt, torch.from_numpy(w).cuda()).cpu().numpy()
                np.testing.assert_array_equal(A, oracle.accumulate_weighted(d, w.astype(np.float64)), err_msg=name)
                assert d8.get_status() == "OK"
    finally:
        d8.set_strategy("ring")
