"""The backward pass at widths that are not multiples of 4, radius 8 above all (its box sums have an
instance of their own there) and eight guides: padded workspace rows, 1 to 3 pixels left for the
last thread of a row, the edges of the 64-column tiles, against the FP64 oracle's analytic
gradient at the bars of test_flr_backward_gpu, whose derivation does not depend on the frame
size or the radius."""
import numpy as np
import pytest

import oracle
import synth
from test_flr_backward_gpu import compare, flr, run_bwd  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,r,rc", [(40, 63, 8, 8), (70, 65, 8, 8), (33, 66, 8, 8), (64, 129, 8, 8), (20, 131, 8, 8), (65, 17, 8, 8),
                                      (48, 130, 8, 0), (37, 61, 5, 8), (37, 62, 8, 5), (30, 127, 5, 5), (21, 67, 3, 2), (1, 19, 8, 8),
                                      (24, 15, 8, 8), (24, 13, 5, 5)])
def test_backward_at_every_kind_of_width(flr, H, W, r, rc):  # noqa: F811
    g, y = synth.random_frame(500 + H + W, H, W, 8)
    G = np.random.default_rng(H * W + r).normal(size=(3, H, W)).astype(np.float32)
    compare(run_bwd(flr, g, y, G, r, rc, 1e-3), oracle.flr_backward(g, y, G, r, 1e-3, coef_radius=rc))


@pytest.mark.parametrize("H,W", [(40, 65), (33, 130), (29, 63)])
def test_backward_separate_map_guide(flr, H, W):  # noqa: F811
    g, y = synth.random_frame(600 + H + W, H, W, 8)
    z, _ = synth.random_frame(601 + H + W, H, W, 8)
    G = np.random.default_rng(H * W).normal(size=(3, H, W)).astype(np.float32)
    compare(run_bwd(flr, g, y, G, 8, 8, 1e-3, z=z), oracle.flr_backward(g, y, G, 8, 1e-3, coef_radius=8, map_guide=z))
