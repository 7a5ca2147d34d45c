"""The backward pass without an eps gradient: its spare slot lies inside the workspace and is
8-byte aligned for every guide count and pixel count (an even number of guides has an odd number of
workspace planes, so with an odd pixel count their end is not), and the other gradients are those
of a call that asks for it."""
import numpy as np
import pytest

import synth
from helpers import to_dev
from test_flr_backward_gpu import flr  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("q", range(1, 9))
@pytest.mark.parametrize("H,W", [(33, 35), (32, 36), (1, 17), (7, 128)])
def test_backward_without_eps_gradient(flr, q, H, W):  # noqa: F811
    import torch
    g, y = synth.random_frame(40 + q, H, W, q)
    G = np.random.default_rng(q).normal(size=(3, H, W)).astype(np.float32)
    f = flr.FLR(q=q, radius=3, coef_radius=2)
    a = f.backward(to_dev(g), to_dev(y), to_dev(G), need_eps=False)
    b = f.backward(to_dev(g), to_dev(y), to_dev(G), need_eps=True)
    torch.cuda.synchronize()
    for k in a:
        assert torch.equal(a[k], b[k]), k
    f.close()
