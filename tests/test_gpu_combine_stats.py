"""The statistics of the last combine after a fill has taken the workspace: one
that grows it, and one that fits and writes over the combine's counters."""
import pytest
import torch

import demgen
from tests.gpu_util import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("strategy", ["ring", "jump"])
def test_stats_after_fill(d8, strategy):
    d = to_dev(demgen.serpentine_dirs(600, 700))
    dev = torch.cuda.current_device()
    kept = d8._ctx.pop(dev, None)  # a context of its own, whose workspace is still small
    try:
        d8.set_strategy(strategy)
        d8.accumulate(d)
        want = d8.combine_stats()
        assert want["top_units"] == 4 and want["top_exits"] > 0
        assert (want["top_jump_rounds"] is None) == (strategy == "ring")
        assert d8.combine_stats() == want
        # a workspace of 22 to 30 bytes a slot is 1.4 to 1.9 a cell, a fill's 0.53:
        # 4096 x 4096 cells are 40 times 600 x 700, 1700 x 1700 seven times
        for side in (4096, 1700):
            z = torch.rand((side, side), device="cuda")
            d8.accumulate(d)
            d8.fill(z)
            assert d8.combine_stats() == want
        assert d8.get_status() == "OK"
    finally:
        d8.set_strategy("ring")
        d8.load().d8_destroy(d8._ctx.pop(dev))
        if kept is not None:
            d8._ctx[dev] = kept
