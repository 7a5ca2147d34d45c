"""The averaging and application of the models at every radius, at the edges of its 64 x 64 tiles
and with padded and unpadded coefficient rows, and the forward kernel at widths whose rows are not
16-byte aligned: against the FP64 oracle at the bar of the other forward tests, and one staging
against the other bit for bit."""
import ctypes

import pytest

import oracle
import synth
from helpers import TOL, rel_err, to_dev
from test_flr_gpu import check, flr  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rc", range(1, 17))
def test_every_coefficient_radius(flr, rc):  # noqa: F811
    H, W, q, r = 62 + rc, 61 + 2 * rc, 3 + rc % 6, 1 + (5 * rc) % 16
    g, y = synth.random_frame(900 + rc, H, W, q)
    check(flr, g, y, r, rc)


@pytest.mark.parametrize("H,W,q,r,rc", [(64, 15, 6, 6, 6), (65, 16, 6, 6, 6), (63, 17, 5, 12, 4), (128, 63, 8, 7, 2),
                                        (129, 65, 3, 2, 16), (1, 97, 4, 3, 3), (130, 1, 4, 3, 3), (64, 1021, 6, 6, 0)])
def test_tile_edges_and_row_padding(flr, H, W, q, r, rc):  # noqa: F811
    g, y = synth.random_frame(1000 + H + W, H, W, q)
    check(flr, g, y, r, rc)


def test_unpadded_rows_equal_padded_rows(flr):  # noqa: F811
    """A 17-column frame of nearly all the pixels of the fixed workspace: its 8-guide models have
    no room for padded rows there, while a handle pads them."""
    import torch
    H, W = 3855, 17
    g, y = synth.random_frame(31, H, W, 8)
    G, Y, out = to_dev(g), to_dev(y), torch.empty((3, H, W), device="cuda")
    params = flr.FlrParams(8, 3, 2, 1e-3, 1e-3, 0)
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    st = flr.load_library().flr_denoise_noalloc(ctypes.byref(params), ptr(G), None, ptr(Y), ptr(out), H, W,
                                                ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    assert st == 0
    f = flr.FLR(q=8, radius=3, coef_radius=2, eps=1e-3, pivot_ratio=1e-3)
    ref = f.denoise(G, Y)
    torch.cuda.synchronize()
    assert torch.equal(out, ref)
    assert rel_err(out.cpu().numpy(), oracle.flr_forward(g, y, 3, 1e-3, coef_radius=2)) <= TOL
    f.close()
