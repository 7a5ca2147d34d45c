"""The guide network's plane and parity layouts and its several-tiles-per-stage kernels against
the NHWC tensors and kernels of flnr_layer: the same products in the same order, so the whole
forward pass equals the chain of its layers bit for bit; and the weight gradients at sizes with
ragged tiles (partial columns, rows and tap columns split over CTAs) against float64 sums."""
import numpy as np
import pytest
import torch
import torch.nn.functional as F

from oracle import flnr_ref
from paper_2410_11625_gb300 import flnr

pytestmark = pytest.mark.gpu


def _net(N, H, W, outputs=8):
    rng = np.random.default_rng(3)
    p = flnr_ref.init_weights(5, outputs)
    for k in p:
        if k.endswith(".b"):
            p[k] = rng.normal(scale=0.1, size=p[k].shape).astype(np.float32)
    return flnr.FLNR(N * H * W, p, outputs=outputs)


@pytest.mark.parametrize("N,H,W", [(1, 4, 4), (2, 20, 36), (1, 132, 268), (3, 128, 128), (1, 544, 804)])
def test_forward_equals_the_chain_of_its_layers(N, H, W):
    net = _net(N, H, W)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(H)
    x = torch.rand((N, 11, H, W), device="cuda", generator=gen) * 2 - 1
    x[:, 8:] = torch.randint(0, 3, (N, 3, H, W), device="cuda", generator=gen).float()  # log1p far from rounding ties
    want = net.forward(x)

    packed = torch.zeros((N, H, W, 16), device="cuda")
    packed[..., :8] = x[:, :8].permute(0, 2, 3, 1)
    packed[..., 8:11] = torch.log1p(x[:, 8:]).permute(0, 2, 3, 1)
    bf = dict(dtype=torch.bfloat16, device="cuda")

    def layer(l, a, h, w, c, b=None, down=1):
        out = torch.empty((N, h // down, w // down, c), **bf)
        return net.layer(l, net.OP_FORWARD, a, b=b, out=out, size=(N, h, w))
    f0 = layer(1, layer(0, packed.to(torch.bfloat16).contiguous(), H, W, 16), H, W, 16)
    f1 = layer(3, layer(2, f0, H, W, 32), H, W, 32, down=2)
    f2 = layer(5, layer(4, f1, H // 2, W // 2, 64), H // 2, W // 2, 64, down=2)
    d1 = layer(7, layer(6, f2, H // 2, W // 2, 32, b=f1), H // 2, W // 2, 32)
    d0 = layer(9, layer(8, d1, H, W, 16, b=f0), H, W, 16)
    a5 = layer(10, d0, H, W, 16)
    got = torch.empty((N, 8, H, W), device="cuda")
    net.layer(11, net.OP_FORWARD, a5, out=got, size=(N, H, W))
    net.status()
    assert torch.equal(got, want)
    net.close()


# Derivation of the bar: products of bfloat16 values are exact in FP32 and at most n = N H W of them
# are accumulated, each addition within 2^-23 of the sum S of their absolute values (as the layer
# tests' bound, no bfloat16 rounding here).
@pytest.mark.parametrize("l", [0, 1, 4, 5, 6, 8])
@pytest.mark.parametrize("N,H,W", [(1, 8, 8), (1, 34, 20), (2, 50, 132)])
def test_weight_gradient_at_ragged_sizes(l, N, H, W):
    net = _net(2 * N, H, W)  # layer 5 spreads its gradient: 64 channels in scratch for 48 per pixel
    name, cin, cout, k = flnr.LAYERS[l]
    cip, cop = -(-cin // 16) * 16, -(-cout // 16) * 16
    s = 2 if l in (3, 5) else 1
    gen = torch.Generator(device="cuda")
    gen.manual_seed(l * 100 + H)
    x = torch.zeros((N, H, W, cip), device="cuda")
    x[..., :cin] = torch.rand((N, H, W, cin), device="cuda", generator=gen) - 0.3
    dz = torch.zeros((N, H // s, W // s, cop), device="cuda")
    dz[..., :cout] = torch.randn((N, H // s, W // s, cout), device="cuda", generator=gen)
    x, dz = x.to(torch.bfloat16).contiguous(), dz.to(torch.bfloat16).contiguous()
    net.zero_grads(x)
    net.layer(l, net.OP_WGRAD, x, b=dz, size=(N, H, W))
    net.status()
    got = flnr.unflatten(net.grads())
    x64 = x.double().cpu().permute(0, 3, 1, 2)[:, :cin]
    z64 = dz.double().cpu().permute(0, 3, 1, 2)[:, :cout]

    def sums(a, z):
        pad = F.pad(a, (k // 2,) * 4)
        return torch.stack([torch.stack([torch.einsum("nihw,nohw->oi", pad[:, :, u:u + H:s, v:v + W:s], z)
                                         for v in range(k)], -1) for u in range(k)], -2)
    n = N * (H // s) * (W // s)
    err = (torch.from_numpy(got[name + ".w"]).double() - sums(x64, z64)).abs()
    assert bool((err <= n * 2.0 ** -23 * sums(x64.abs(), z64.abs()) + 1e-30).all())
    berr = (torch.from_numpy(got[name + ".b"]).double() - z64.sum(dim=(0, 2, 3))).abs()
    assert bool((berr <= n * 2.0 ** -23 * z64.abs().sum(dim=(0, 2, 3))).all())
    net.close()
