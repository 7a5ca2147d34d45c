"""The backward pass's tiled box sums at the edges of their 64 x 64 tiles and at each kind of
radius (8 and 5 compiled in, others at run time, up to the largest), against the FP64 oracle's
analytic gradient at the bars of test_flr_backward_gpu, whose derivation does not depend on the
frame size or the radius."""
import numpy as np
import pytest

import oracle
import synth
from test_flr_backward_gpu import compare, flr, run_bwd  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,r,rc", [(64, 64, 8, 8), (65, 68, 8, 5), (63, 60, 5, 8), (72, 132, 5, 5), (129, 124, 3, 4),
                                      (66, 128, 16, 16), (8, 4, 8, 1), (1, 8, 5, 5), (130, 64, 1, 2)])
def test_box_sums_at_tile_edges(flr, H, W, r, rc):  # noqa: F811
    g, y = synth.random_frame(700 + H + r, H, W, 8)
    G = np.random.default_rng(H * W + r).normal(size=(3, H, W)).astype(np.float32)
    compare(run_bwd(flr, g, y, G, r, rc, 1e-3), oracle.flr_backward(g, y, G, r, 1e-3, coef_radius=rc))
