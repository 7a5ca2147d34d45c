"""The network's backward pass in its own forms -- plane and parity layouts, several row phases per
stage, the strided weight gradients on parity planes, the concatenated decoder inputs -- against the
chain of its layers by themselves (flnr_layer: NHWC tensors): the gradient of every layer's output
comes from the same products in the same order, so it is known bit for bit, and the weight and
bias gradients are compared with float64 sums of those very values.

Bar of the weight gradients, per element, in units of S = sum |x dz|: two tiles of 128 pixels are
accumulated by the tensor cores, 16 instructions that may each lose two units in the last place
(2 x 2^-23), and at most 64 FP32 additions of partial sums follow (2^-24 each) on these sizes.
Bias gradients: the additions alone (8 + 7 within a tile, 6 across lanes, then as above: 2^-24 x 96).
"""
import numpy as np
import pytest
import torch
import torch.nn.functional as F

from oracle import flnr_ref
from paper_2410_11625_gb300 import flnr

pytestmark = pytest.mark.gpu

W_TOL = 16 * 2 * 2.0 ** -23 + 64 * 2.0 ** -24
B_TOL = 96 * 2.0 ** -24


def _net(N, H, W):
    rng = np.random.default_rng(3)
    p = flnr_ref.init_weights(5, 8)
    for k in p:
        if k.endswith(".b"):
            p[k] = rng.normal(scale=0.1, size=p[k].shape).astype(np.float32)
    return flnr.FLNR(N * H * W, p, outputs=8)


def sums(x, dz, cin, cout, k, s):
    """float64 sums of the weight gradient and of its absolute values, and the same of the bias."""
    N, H, W = x.shape[:3]
    ref = torch.zeros((cout, cin, k, k), dtype=torch.float64, device=x.device)
    mag = torch.zeros_like(ref)
    for n in range(N):
        a = F.pad(x[n, ..., :cin].double().permute(2, 0, 1), (k // 2,) * 4)
        z = dz[n, ..., :cout].double().permute(2, 0, 1).reshape(cout, -1)
        for u in range(k):
            for v in range(k):
                m = a[:, u:u + H:s, v:v + W:s].reshape(cin, -1)
                ref[:, :, u, v] += z @ m.T
                mag[:, :, u, v] += z.abs() @ m.abs().T
    b = dz[..., :cout].double().sum((0, 1, 2))
    return ref, mag, b, dz[..., :cout].double().abs().sum((0, 1, 2))


@pytest.mark.parametrize("N,H,W", [(1, 4, 4), (1, 36, 20), (3, 132, 140), (2, 268, 396)])
def test_backward_equals_the_chain_of_its_layers(N, H, W):
    net = _net(N, H, W)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(H)
    x = torch.rand((N, 11, H, W), device="cuda", generator=gen) * 2 - 1
    x[:, 8:] = torch.randint(0, 3, (N, 3, H, W), device="cuda", generator=gen).float()
    go = torch.randn((N, 8, H, W), device="cuda", generator=gen)
    bf = dict(dtype=torch.bfloat16, device="cuda")
    h2, w2, h4, w4 = H // 2, W // 2, H // 4, W // 4

    def fwd(l, a, h, w, c, b=None, down=1):
        out = torch.empty((N, h // down, w // down, c), **bf)
        return net.layer(l, net.OP_FORWARD, a, b=b, out=out, size=(N, h, w))

    def dgrad(l, dz, h, w, c, mask=None):
        return net.layer(l, net.OP_DGRAD, dz, mask=mask, out=torch.empty((N, h, w, c), **bf), size=(N, h, w))

    def up(t):
        return t.repeat_interleave(2, 1).repeat_interleave(2, 2)

    def down_sum(g, mask):  # the 2 x 2 sum of the upsampling's adjoint, through the ReLU
        f = g.float()
        s = ((f[:, ::2, ::2] + f[:, ::2, 1::2]) + f[:, 1::2, ::2]) + f[:, 1::2, 1::2]
        return torch.where(mask > 0, s, 0.0).to(torch.bfloat16).contiguous()

    def join(skip, path, mask):
        return torch.where(mask > 0, path.float() + skip, 0.0).to(torch.bfloat16).contiguous()

    packed = torch.zeros((N, H, W, 16), device="cuda")
    packed[..., :8] = x[:, :8].permute(0, 2, 3, 1)
    packed[..., 8:11] = torch.log1p(x[:, 8:]).permute(0, 2, 3, 1)
    x0 = packed.to(torch.bfloat16).contiguous()
    a0 = fwd(0, x0, H, W, 16)
    f0 = fwd(1, a0, H, W, 16)
    a1 = fwd(2, f0, H, W, 32)
    f1 = fwd(3, a1, H, W, 32, down=2)
    a2 = fwd(4, f1, h2, w2, 64)
    f2 = fwd(5, a2, h2, w2, 64, down=2)
    a3 = fwd(6, f2, h2, w2, 32, b=f1)
    d1 = fwd(7, a3, h2, w2, 32)
    a4 = fwd(8, d1, H, W, 16, b=f0)
    d0 = fwd(9, a4, H, W, 16)
    a5 = fwd(10, d0, H, W, 16)
    s = torch.empty((N, 8, H, W), device="cuda")
    net.layer(11, net.OP_FORWARD, a5, out=s, size=(N, H, W))
    dz = [None] * 12
    head = torch.zeros((N, H, W, 16), device="cuda")
    head[..., :8] = (go * s * (1.0 - s)).permute(0, 2, 3, 1)
    dz[11] = head.to(torch.bfloat16).contiguous()
    dz[10] = dgrad(11, dz[11], H, W, 16, a5)
    dz[9] = dgrad(10, dz[10], H, W, 16, d0)
    dz[8] = dgrad(9, dz[9], H, W, 16, a4)
    g = dgrad(8, dz[8], H, W, 48)
    dz[7], skip0 = down_sum(g[..., :32], d1), g[..., 32:].float()
    dz[6] = dgrad(7, dz[7], h2, w2, 32, a3)
    g = dgrad(6, dz[6], h2, w2, 96)
    dz[5], skip1 = down_sum(g[..., :64], f2), g[..., 64:].float()
    dz[4] = dgrad(5, dz[5], h2, w2, 64, a2)
    dz[3] = join(skip1, dgrad(4, dz[4], h2, w2, 32), f1)
    dz[2] = dgrad(3, dz[3], H, W, 32, a1)
    dz[1] = join(skip0, dgrad(2, dz[2], H, W, 16), f0)
    dz[0] = dgrad(1, dz[1], H, W, 16, a0)
    want_in = dgrad(0, dz[0], H, W, 16).float()[..., :11].permute(0, 3, 1, 2)

    assert torch.equal(net.forward(x), s)
    gi = torch.empty_like(x)
    net.zero_grads(x)
    net.backward(go, grad_in=gi)
    net.status()
    got = flnr.unflatten(net.grads())
    # the guides' gradients to the bit; the radiance's within the rounding of exp(-L) and its product
    assert torch.equal(gi[:, :8], want_in[:, :8])
    L = x0[..., 8:11].float().permute(0, 3, 1, 2)
    want_rad = torch.where(L > 0, want_in[:, 8:] * torch.exp(-L), 0.0)
    assert bool(((gi[:, 8:] - want_rad).abs() <= 8 * 2.0 ** -24 * want_rad.abs()).all())
    xs = [x0, a0, f0, a1, f1, a2, torch.cat([up(f2), f1], -1), a3, torch.cat([up(d1), f0], -1), a4, d0, a5]
    for l, (name, cin, cout, k) in enumerate(flnr.LAYERS):
        ref, mag, b, bmag = sums(xs[l], dz[l], cin, cout, k, 2 if l in (3, 5) else 1)
        err = (torch.from_numpy(np.ascontiguousarray(got[name + ".w"])).cuda().double() - ref).abs()
        assert bool((err <= W_TOL * mag + 1e-30).all()), (name, float((err / (mag + 1e-30)).max()))
        berr = (torch.from_numpy(np.ascontiguousarray(got[name + ".b"])).cuda().double() - b).abs()
        assert bool((berr <= B_TOL * bmag + 1e-30).all()), (name, float((berr / (bmag + 1e-30)).max()))
    net.close()


@pytest.mark.parametrize("l", [0, 1, 4, 8])
def test_weight_gradients_do_not_lose_bits_with_the_frame_size(l):
    """Operands of one sign on a 1920x1080 frame, where a running sum of the tensor cores, which do
    not round to nearest, falls behind by a unit with every instruction: 6.5e-5 of the sum when a
    CTA's 860 instructions were one chain.  Bar: as above, with the 54 sums of a CTA's 107 tiles and
    the reduction's 26 more among the FP32 additions."""
    net = _net(2, 1080, 1920)
    name, cin, cout, k = flnr.LAYERS[l]
    cip, cop = -(-cin // 16) * 16, -(-cout // 16) * 16
    gen = torch.Generator(device="cuda")
    gen.manual_seed(l)
    x = torch.zeros((1, 1080, 1920, cip), device="cuda")
    x[..., :cin] = torch.rand((1, 1080, 1920, cin), device="cuda", generator=gen) + 0.25
    dz = torch.zeros((1, 1080, 1920, cop), device="cuda")
    dz[..., :cout] = torch.rand((1, 1080, 1920, cout), device="cuda", generator=gen)
    x, dz = x.to(torch.bfloat16).contiguous(), dz.to(torch.bfloat16).contiguous()
    net.zero_grads(x)
    net.layer(l, net.OP_WGRAD, x, b=dz, size=(1, 1080, 1920))
    net.status()
    got = torch.from_numpy(np.ascontiguousarray(flnr.unflatten(net.grads())[name + ".w"])).cuda().double()
    ref, mag, _, _ = sums(x, dz, cin, cout, k, 1)
    rel = float(((got - ref).abs() / mag).max())
    assert rel <= 16 * 2 * 2.0 ** -23 + (54 + 26) * 2.0 ** -24, rel
    net.close()
