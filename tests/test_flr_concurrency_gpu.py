"""flr_set_concurrency changes only the split of the work: every share of the device gives a result
that meets the FP64 oracle at the bars of the forward and backward tests, handles of one share run
side by side on their own streams, and bad values are refused."""
import numpy as np
import pytest

import oracle
import synth
from helpers import TOL, rel_err, to_dev
from test_flr_backward_gpu import compare, flr  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 3, 16, 152, 1000])
@pytest.mark.parametrize("q,r,rc,H,W", [(8, 8, 8, 128, 128), (8, 5, 5, 37, 84), (6, 4, 3, 70, 101)])
def test_share_of_the_device(flr, n, q, r, rc, H, W):  # noqa: F811
    import torch
    frames, streams = [], [torch.cuda.Stream() for _ in range(3)]
    for k, s in enumerate(streams):
        g, y = synth.random_frame(50 + k, H, W, q)
        G = np.random.default_rng(k).normal(size=(3, H, W)).astype(np.float32)
        f = flr.FLR(q=q, radius=r, coef_radius=rc, eps=1e-3)
        f.set_concurrency(n)
        f.reserve(H, W)
        frames.append((f, g, y, G, to_dev(g), to_dev(y), to_dev(G)))
    torch.cuda.synchronize()
    res = []
    for s, (f, _, _, _, g, y, G) in zip(streams, frames):
        with torch.cuda.stream(s):
            res.append((f.denoise(g, y), f.backward(g, y, G, need_eps=True)))
    torch.cuda.synchronize()
    for (f, g, y, G, *_), (out, grad) in zip(frames, res):
        assert rel_err(out.cpu().numpy(), oracle.flr_forward(g, y, r, 1e-3, coef_radius=rc)) <= TOL
        got = {k: v.cpu().numpy().astype(np.float64) for k, v in grad.items()}
        got["eps"] = float(got["eps"][0])
        compare(got, oracle.flr_backward(g, y, G, r, 1e-3, coef_radius=rc))
        f.close()


def test_bad_values_are_refused(flr):  # noqa: F811
    f = flr.FLR(q=8)
    for n in (0, -1):
        with pytest.raises(flr.FlrError):
            f.set_concurrency(n)
    f.close()
