"""The averaging and application of eight guides' models, three colours together (coefficient radii up
to 12, padded rows): at the edges of its 64 x 32 tiles and in row bands against the FP64 oracle, bit for
bit against the general form that unpadded rows take, and no slower than seven guides, whose eight
planes a colour take the general form."""
import ctypes

import numpy as np
import pytest

import oracle
import synth
from helpers import TOL, rel_err, to_dev
from test_flr_gpu import check, flr  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,r,rc", [(32, 64, 5, 8), (31, 63, 8, 5), (33, 65, 5, 8), (64, 16, 2, 12), (1, 130, 4, 8),
                                      (97, 18, 3, 1), (65, 127, 1, 7), (8, 129, 6, 4), (70, 65, 3, 13)])
def test_tile_edges(flr, H, W, r, rc):  # noqa: F811
    g, y = synth.random_frame(1300 + H + W, H, W, 8)
    check(flr, g, y, r, rc)


@pytest.mark.parametrize("rc", [1, 3, 4, 5, 8, 9, 12, 13])
def test_equals_the_general_form(flr, rc):  # noqa: F811
    """17 columns of nearly all the pixels of the fixed workspace, which has no room for padded rows."""
    import torch
    H, W = 3855, 17
    g, y = synth.random_frame(50 + rc, H, W, 8)
    G, Y, out = to_dev(g), to_dev(y), torch.empty((3, H, W), device="cuda")
    params = flr.FlrParams(8, 3, rc, 1e-3, 1e-3, 0)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    st = flr.load_library().flr_denoise_noalloc(ctypes.byref(params), ptr(G), None, ptr(Y), ptr(out), H, W,
                                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    f = flr.FLR(q=8, radius=3, coef_radius=rc, eps=1e-3, pivot_ratio=1e-3)
    ref = f.denoise(G, Y)
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    f.close()


@pytest.mark.parametrize("H,W,r,rc", [(203, 70, 5, 8), (131, 257, 8, 5)])
def test_row_bands(flr, H, W, r, rc):  # noqa: F811
    g, y = synth.random_frame(1400 + H, H, W, 8)
    f = flr.FLR(q=8, radius=r, coef_radius=rc, eps=1e-3, pivot_ratio=1e-3)
    out = f.denoise_host(np.ascontiguousarray(g, np.float32), np.ascontiguousarray(y, np.float32))
    assert rel_err(out, oracle.flr_forward(g, y, r, 1e-3, coef_radius=rc)) <= TOL
    f.close()


@pytest.mark.parametrize("r,rc", [(5, 8), (8, 5)])
def test_no_slower_than_seven_guides(flr, r, rc):  # noqa: F811
    """27 planes together against 24 one colour after the other: 29 and 35 us at rc = 5 (39 us for the
    27 one colour after the other)."""
    import torch
    us = {}
    for q in (7, 8):
        g, y = synth.random_frame(7, 480, 640, q)
        G, Y = to_dev(g), to_dev(y)
        f = flr.FLR(q=q, radius=r, coef_radius=rc, timing=True)
        runs = []
        for _ in range(7):
            for _ in range(10):
                f.denoise(G, Y)
            torch.cuda.synchronize()
            runs.append(f.kernel_times()["apply_ms"] * 100)
        us[q] = sorted(runs[2:])[2]
        f.close()
    assert us[8] <= us[7], us
