"""The fill with and without the coarser grids on grids that have them, as d8_fill
calls it where device memory has and has not room for them (the library's own
run_fill, by its linker name): the same bits, and those of the oracle."""
import ctypes

import numpy as np
import pytest
import torch

import demgen
import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(577, 643), (640, 1500), (1300, 1100)])
def test_fill_starts(d8, shape):
    H, W = shape
    L = d8.load()
    i64, vp, i32 = ctypes.c_int64, ctypes.c_void_p, ctypes.c_int
    ws_bytes, run = L._ZN2d813fill_ws_bytesEllb, L._ZN2d88run_fillEPKflllfPflPvbPjP11CUstream_stlPlPbPi
    ws_bytes.argtypes, ws_bytes.restype = [i64, i64, ctypes.c_bool], ctypes.c_size_t
    run.argtypes = [vp, i64, i64, i64, ctypes.c_float, vp, i64, vp, ctypes.c_bool, vp, vp, i64, vp, vp, vp]
    assert ws_bytes(H, W, True) > H * W // 2 > ws_bytes(H, W, False)
    rng = np.random.default_rng(H)
    channel = demgen.serpentine_dem(H | 1, W)[:H].copy()
    channel[H // 2, W // 2] = channel.max()
    for name, z in (("fractal", demgen.fractal_raw(H, W, seed=H)), ("dam", channel),
                    ("pits", (rng.integers(-3, 4, size=shape) * 0.5).astype(np.float32))):
        ref = oracle.fill_eps(z, 1e-3)
        zt = torch.from_numpy(z).cuda()
        for coarse in (True, False):
            F = torch.full((H, W), -9.0, device="cuda")
            ws = torch.empty(ws_bytes(H, W, coarse), dtype=torch.uint8, device="cuda")
            status = torch.zeros(1, dtype=torch.int32, device="cuda")
            rounds, timed_out, launches = i64(), ctypes.c_bool(), i32()
            assert run(zt.data_ptr(), H, W, W, 1e-3, F.data_ptr(), W, ws.data_ptr(), coarse, status.data_ptr(),
                       torch.cuda.current_stream().cuda_stream, 1 << 20, ctypes.byref(rounds), ctypes.byref(timed_out),
                       ctypes.byref(launches)) == 0
            assert not timed_out.value and int(status.item()) == 0
            np.testing.assert_array_equal(F.cpu().numpy(), ref, err_msg=f"{name} {coarse}")
