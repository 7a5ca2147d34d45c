"""Frames of which about half the pixels are flagged, in pairs of neighbours with one, both or none
flagged: the packed solve leaves the right one out, the lists run in (row, column) order and the
FP64 shares come back.  The threshold is the median of the float64 pivot ratios of the frame itself.
Bar: the parity metric's, as for every uniform frame."""
import numpy as np
import pytest

import oracle
import synth
from helpers import TOL, rel_err
from test_flr_fused_gpu import flr, run  # noqa: F401

pytestmark = pytest.mark.gpu


def pivot_ratios(g, r, eps):
    """Smallest Cholesky pivot ratio d_j / M_jj of every pixel's centred, ridged moment matrix."""
    q, H, W = g.shape
    g = g.astype(np.float64) - g.mean(axis=(1, 2), keepdims=True)

    def box(a):
        c = np.zeros(a.shape[:-2] + (H + 1, W + 1))
        c[..., 1:, 1:] = a.cumsum(-2).cumsum(-1)
        y0, y1 = np.maximum(np.arange(H) - r, 0), np.minimum(np.arange(H) + r, H - 1) + 1
        x0, x1 = np.maximum(np.arange(W) - r, 0), np.minimum(np.arange(W) + r, W - 1) + 1
        s = c[..., y1, :] - c[..., y0, :]
        return s[..., x1] - s[..., x0]
    n = box(np.ones((H, W)))
    mu = box(g) / n
    M = box(g[:, None] * g[None]) / n - mu[:, None] * mu[None] + eps * np.eye(q)[:, :, None, None]
    M = np.moveaxis(M, (0, 1), (2, 3))
    L = np.linalg.cholesky(M)
    d = np.diagonal(L, axis1=2, axis2=3) ** 2
    return (d / np.diagonal(M, axis1=2, axis2=3)).min(-1)


@pytest.mark.parametrize("H,W,r,rc", [(65, 92, 8, 0), (43, 164, 8, 8), (33, 88, 5, 5), (50, 200, 8, 8), (21, 60, 5, 5), (24, 196, 8, 0)])
def test_half_of_the_pixels_flagged(flr, H, W, r, rc):  # noqa: F811
    g, y = synth.random_frame(H * 11 + W, H, W, 8)
    ratio = pivot_ratios(g, r, 1e-3)
    tau = float(np.float32(np.median(ratio)))
    low = ratio <= tau
    # pairs as the solver takes them: from column x0 - rc of a strip, x0 even
    at = np.pad(low, ((0, 0), (rc & 1, 1)))
    pairs = at[:, : (W + 1) // 2 * 2].reshape(H, -1, 2).sum(-1)
    assert (pairs == 1).any() and (pairs == 2).any() and (pairs == 0).any()
    got, st = run(flr, g, y, r, rc, pivot_ratio=tau)
    # FP32 pivots differ from the float64 ones by their rounding
    near = int((np.abs(ratio - tau) < 1e-4).sum())
    assert abs(st["flagged"] - int(low.sum())) <= near < H * W // 4
    assert 0 < st["flagged"] < H * W and st["resolved"] == st["flagged"]
    assert np.all(np.isfinite(got))
    assert rel_err(got, oracle.flr_forward(g, y, r, 1e-3, coef_radius=rc)) <= TOL
    again, st2 = run(flr, g, y, r, rc, pivot_ratio=tau)
    assert np.array_equal(got, again) and st2["flagged"] == st["flagged"]
