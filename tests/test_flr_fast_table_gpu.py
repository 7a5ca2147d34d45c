"""Batches of the fast path whose frames take different last stages (16-byte aligned rows, odd
rows, cells above 8 pixels): each frame equals its own call bit for bit, and the flagged blocks
of a batch are the sum over its frames."""
import pytest

import synth
from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def flr():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2410_11625_gb300 import flr as mod
    return mod


@pytest.mark.parametrize("q,factor,scale,sizes", [
    (8, 8, 1, [(1, 1), (8, 512), (9, 516), (64, 1023), (17, 130), (33, 132)]),
    (8, 4, 2, [(31, 33), (32, 34), (5, 6)]),
    (4, 2, 1, [(10, 1026), (7, 3)]),
    (1, 8, 2, [(24, 40), (23, 41)]),          # cells of 16 pixels: no frame takes the tiled apply
    (8, 8, 1, [(16 + k, 40 + 3 * k) for k in range(16)])])
def test_mixed_batch_equals_single_frames(flr, q, factor, scale, sizes):
    import torch
    f = flr.FastFLR(q=q, factor=factor, scale=scale, eps=1e-5, pivot_ratio=1e-2)
    frames, single, flagged = [], [], 0
    for k, (H, W) in enumerate(sizes):
        g, y = synth.random_frame(100 + k, H, W, q)
        z, _ = synth.random_frame(200 + k, H * scale, W * scale, q)
        frames.append((to_dev(g), to_dev(y), to_dev(z), torch.full((3, H * scale, W * scale), float("nan"), device="cuda")))
    for g, y, z, _ in frames:
        single.append(f.denoise(g, y, map_guide=z).clone())
        flagged += f.stats()["flagged"]
    for _ in range(2):
        f.denoise_batch(frames)
        assert f.batch_status() == 0
        assert f.stats()["flagged"] == flagged
        for (_, _, _, o), s in zip(frames, single):
            assert torch.equal(o, s)
            o.fill_(float("nan"))
    f.close()
