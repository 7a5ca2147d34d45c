"""The last stage's plain form (cells of more than 8 pixels, rows that do not start on 16-byte
boundaries, parameter gradients at every cell size).  Cells of P = factor * scale pixels begin at
column P r - P/2, a 16-byte boundary only where P is a multiple of 8: cells of 4, 12, 20 and 28 on
output rows that are 16-byte aligned themselves, and cells of up to 64 rows with odd widths at every
guide count, against the FP64 oracle at the bars of test_flr_fast_gpu, whose derivation does
not depend on P; a batch of such frames equals the single calls bit for bit, and frames of odd
width cost about what aligned ones do."""
import numpy as np
import pytest

import oracle
import synth
from helpers import to_dev
from test_flr_fast_gpu import check, flr  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("factor,scale,H,W", [(4, 3, 60, 100), (2, 6, 31, 52), (4, 5, 40, 64), (4, 7, 25, 40), (8, 3, 32, 48)])
def test_wide_cells(flr, factor, scale, H, W):  # noqa: F811
    g, y = synth.render(4, H, W)
    z, _ = synth.render(4, H * scale, W * scale)
    check(flr, g, y, z=z, scale=scale, factor=factor, rms_bar=True)


@pytest.mark.parametrize("factor,scale,H,W", [(2, 1, 49, 80), (4, 1, 40, 260), (2, 2, 33, 62), (2, 3, 20, 128)])
def test_small_cells(flr, factor, scale, H, W):  # noqa: F811
    """Cells of 2, 4 and 6 pixels in the tiled form."""
    g, y = synth.random_frame(40 + H, H, W, 8)
    z = synth.random_frame(41 + H, H * scale, W * scale, 8)[0] if scale > 1 else None
    check(flr, g, y, z=z, scale=scale, factor=factor, rms_bar=scale > 1)


@pytest.mark.parametrize("factor,scale,H,W", [(4, 1, 96, 160), (2, 2, 48, 80), (4, 3, 32, 48), (2, 1, 49, 80)])
def test_parameter_gradients(flr, factor, scale, H, W):  # noqa: F811
    import torch
    g, y = synth.render(12, H, W)
    z = synth.render(12, H * scale, W * scale)[0] if scale > 1 else None
    kw = dict(factor=factor, sigma_blocks=1.1, taps=3, eps=2e-3, map_guide=z, scale=scale)
    out = oracle.flr_fast(g, y, **kw)
    G = (out - 0.9 * np.mean(out, axis=(1, 2), keepdims=True)).astype(np.float32)
    ref = oracle.flr_fast_param_grads(g, y, G, **kw)
    f = flr.FastFLR(q=8, factor=factor, scale=scale, sigma=1.1, taps=3, eps=2e-3)
    got = f.param_grad(to_dev(g), to_dev(y), to_dev(G), map_guide=None if z is None else to_dev(z))
    torch.cuda.synchronize()
    got = got.cpu().numpy()
    f.close()
    for t, name in enumerate(["sigma", "eps"]):
        assert abs(got[t] - ref[name]) <= 1e-4 * abs(ref[name]), (name, got[t], ref[name])


@pytest.mark.parametrize("q,factor,scale,H,W", [(1, 8, 2, 9, 33), (2, 8, 3, 17, 20), (3, 4, 4, 10, 43), (4, 8, 1, 20, 129),
                                                (5, 8, 8, 9, 11), (6, 2, 1, 33, 257), (7, 4, 1, 21, 131), (8, 8, 4, 1, 1)])
def test_guide_counts_and_odd_widths(flr, q, factor, scale, H, W):  # noqa: F811
    g, y = synth.random_frame(300 + q, H, W, q)
    z = synth.random_frame(310 + q, H * scale, W * scale, q)[0] if scale > 1 else None
    check(flr, g, y, z=z, scale=scale, factor=factor, rms_bar=True)


def test_batch_of_wide_cells(flr):  # noqa: F811
    import torch
    f = flr.FastFLR(q=8, factor=4, scale=3)
    frames = []
    for k, (H, W) in enumerate([(20, 36), (17, 40), (23, 37)]):
        g, y = synth.random_frame(60 + k, H, W, 8)
        z, _ = synth.random_frame(70 + k, 3 * H, 3 * W, 8)
        frames.append((to_dev(g), to_dev(y), to_dev(z), torch.full((3, 3 * H, 3 * W), float("nan"), device="cuda")))
    f.denoise_batch(frames)
    assert f.batch_status() == 0
    for g, y, z, o in frames:
        assert torch.equal(f.denoise(g, y, map_guide=z), o)
    f.close()


def test_odd_width_costs_about_an_aligned_one(flr):  # noqa: F811
    """Four 1080 x 1919 frames against four 1080 x 1920 ones: the same work and, but for the ends
    of the rows, the same bytes.  0.250 against 0.209 ms (0.477 with one thread per run of 8 pixels
    of a row)."""
    import torch
    f = flr.FastFLR(q=8, factor=8, scale=1)

    def best(W):
        frames = []
        for k in range(4):
            g, y = torch.rand((8, 1080, W), device="cuda"), torch.rand((3, 1080, W), device="cuda")
            frames.append((g, y, g, torch.empty_like(y)))
        times = []
        for _ in range(12):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(5):
                f.denoise_batch(frames)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) / 5)
        return min(times)
    aligned, odd = best(1920), best(1919)
    print(f"aligned {aligned:.4f} ms, odd {odd:.4f} ms")
    assert odd <= 2.0 * aligned
    f.close()
