"""Performance cases of the library: the work its users have it do, through its public
entry points, from one 256 x 256 frame to a 4K frame, a training step and a serving batch.

listed() names the cases, draw(rng) gives further ones of the same ranges, prepare() makes
what a user's program holds before the call, run() is one pass, work() the bytes and
operations a pass cannot do without, and exact() the same results in float64 from plain
PyTorch.  Inputs are procedural rooms (flat albedos, walls, boxes and spheres, a noisy
ambient occlusion, one-sample radiance with a heavy tail), as the renderer in front of the
denoiser gives them.
"""
import math
import random

import numpy as np
import torch
import torch.nn.functional as F

EPS, TAU = 1e-3, 1e-3                 # ridge term and pivot ratio: the benchmark's values
SIGMA, TAPS = 1.25, 3                 # fast FLR's Gaussian, in blocks
LR, BETA1, BETA2, ADAM_EPS, ADAM_T = 1e-3, 0.9, 0.999, 1e-8, 1000
ADAM_RMS = 1e-3                       # root of Adam's second moments in a running training
LAYERS = [("in0", 11, 16, 3), ("in1", 16, 16, 1), ("e1a", 16, 32, 3), ("e1b", 32, 32, 3),
          ("e2a", 32, 64, 3), ("e2b", 64, 64, 3), ("d1a", 96, 32, 3), ("d1b", 32, 32, 3),
          ("d0a", 48, 16, 3), ("d0b", 16, 16, 3), ("o0", 16, 16, 3), ("o1", 16, 8, 1)]


def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def listed():
    return [
        # one small frame at a time: a preview or an interactive viewport (the 256 x 256 workload)
        {"name": "flr_256_r5", "kind": "flr", "H": 256, "W": 256, "q": 8, "r": 5, "rc": 5, "map": False},
        # the headline: one full-HD frame, models averaged over the window
        {"name": "flr_1080p_r8", "kind": "flr", "H": 1080, "W": 1920, "q": 8, "r": 8, "rc": 8, "map": False},
        # a 4K frame with the paper's own reading, every pixel's own model (no averaging)
        {"name": "flr_4k_unaveraged", "kind": "flr", "H": 2160, "W": 3840, "q": 8, "r": 8, "rc": 0, "map": False},
        # six guides (no depth, no occlusion) on a viewport of odd width: the general path
        {"name": "flr_q6_odd", "kind": "flr", "H": 719, "W": 1277, "q": 6, "r": 6, "rc": 6, "map": False},
        # gradients of a full-HD frame: learning through the denoiser
        {"name": "backward_1080p", "kind": "backward", "H": 1080, "W": 1920, "q": 8, "r": 8, "rc": 8, "map": False},
        # one training crop with separate model and map guides, forward and backward by autograd
        {"name": "autograd_crop_map", "kind": "autograd", "H": 128, "W": 128, "q": 8, "r": 8, "rc": 8, "map": True},
        # the paper's fast FLR on a full-HD frame
        {"name": "fast_1080p", "kind": "fast", "H": 1080, "W": 1920, "factor": 8, "scale": 1},
        # joint denoising and 2x upsampling to 2560 x 1440
        {"name": "upsample_1440p", "kind": "fast", "H": 720, "W": 1280, "factor": 4, "scale": 2},
        # the guide network on a full-HD frame (inference)
        {"name": "flnr_forward_1080p", "kind": "flnr_forward", "N": 1, "H": 1080, "W": 1920, "outputs": 8},
        # the guide network's gradients on the training batch, for a user's own optimiser
        {"name": "flnr_grads_16x128", "kind": "flnr_grads", "N": 16, "H": 128, "W": 128, "outputs": 8},
        # one training step: network, denoiser, loss, both adjoints, Adam
        {"name": "train_step_16x128", "kind": "train", "N": 16, "H": 128, "W": 128, "outputs": 8, "loss": "l1"},
        # a serving batch of 8 frames of three sizes, 2x upsampled, with the guide network
        {"name": "serving_8_frames", "kind": "serving", "n0": 3, "n1": 3, "n2": 2, "H": 1080, "W": 1920},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["flr", "flr", "flr_general", "backward", "autograd", "fast", "fast", "flnr_forward",
                       "flnr_grads", "train", "serving"])
    if kind == "flr":  # the radii with one fused kernel, any frame from a tile to 4K
        r, rc = rng.choice([(8, 8), (8, 8), (5, 5), (8, 0)])
        return {"kind": "flr", "H": _log(rng, 96, 2160), "W": 4 * _log(rng, 24, 960), "q": 8, "r": r, "rc": rc,
                "map": rng.random() < 0.25}
    if kind == "flr_general":  # other guide counts, radii and odd widths
        r = rng.randint(2, 12)
        return {"kind": "flr", "H": _log(rng, 96, 1080), "W": _log(rng, 96, 1920), "q": rng.randint(3, 8), "r": r,
                "rc": rng.choice([0, r, max(1, r // 2)]), "map": rng.random() < 0.25}
    if kind == "backward":  # the radii of the two single-frame workloads, any width
        r = rng.choice([8, 8, 5])
        return {"kind": "backward", "H": _log(rng, 96, 1080), "W": _log(rng, 96, 1920), "q": 8, "r": r, "rc": r,
                "map": False}
    if kind == "autograd":
        return {"kind": "autograd", "H": _log(rng, 64, 512), "W": 4 * _log(rng, 16, 128), "q": 8, "r": 8, "rc": 8,
                "map": rng.random() < 0.5}
    if kind == "fast":
        factor, scale = rng.choice([(8, 1), (8, 1), (4, 1), (4, 2), (8, 2)])
        return {"kind": "fast", "H": _log(rng, 128, 2160 // scale), "W": _log(rng, 128, 3840 // scale),
                "factor": factor, "scale": scale}
    if kind == "flnr_forward":
        return {"kind": "flnr_forward", "N": 1, "H": 4 * _log(rng, 32, 270), "W": 4 * _log(rng, 32, 480),
                "outputs": rng.choice([8, 16])}
    if kind in ("flnr_grads", "train"):
        s = {"kind": kind, "N": rng.randint(4, 16), "H": 4 * rng.randint(16, 32), "W": 0, "outputs": rng.choice([8, 16])}
        s["W"] = s["H"]
        if kind == "train":
            s["loss"] = rng.choice(["l1", "smape"])
        return s
    return {"kind": "serving", "n0": rng.randint(1, 3), "n1": rng.randint(1, 2), "n2": rng.randint(0, 1),
            "H": 24 * _log(rng, 8, 45), "W": 24 * _log(rng, 10, 80)}


# ---- inputs --------------------------------------------------------------------------------
def _room(seed, H, W):
    """One frame: guides [8, H, W] (albedo, normal, depth, occlusion), one-sample radiance
    [3, H, W] and the noise-free radiance, float32."""
    rnd, dev = random.Random(seed), _dev()
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    cam = torch.tensor([rnd.uniform(2, 6), rnd.uniform(1, 3), rnd.uniform(0.3, 1.5)], device=dev)
    yaw = rnd.uniform(-0.5, 0.5)
    v = (torch.arange(H, device=dev) + 0.5 - H / 2) / (H / 2) * math.tan(math.pi / 6)
    u = (torch.arange(W, device=dev) + 0.5 - W / 2) / (H / 2) * math.tan(math.pi / 6)
    v, u = torch.meshgrid(v, u, indexing="ij")
    inv = torch.rsqrt(1 + u * u + v * v)
    d = torch.stack([(u * math.cos(yaw) + math.sin(yaw)) * inv, -v * inv, (math.cos(yaw) - u * math.sin(yaw)) * inv])
    d = torch.where(d.abs() < 1e-6, torch.full_like(d, 1e-6), d)
    room = torch.tensor([8.0, 4.0, 8.0], device=dev)
    far = torch.where(d > 0, (room - cam)[:, None, None], cam[:, None, None]) / d.abs()
    t, axis = far.min(dim=0)  # the wall the ray leaves the room through
    obj = 2 * axis + (d.gather(0, axis[None])[0] > 0).long()
    n = torch.zeros_like(d).scatter_(0, axis[None], -torch.sign(d.gather(0, axis[None])))
    for k in range(8):  # boxes
        lo = torch.tensor([rnd.uniform(0, 7), rnd.uniform(0, 2), rnd.uniform(2.5, 7)], device=dev)
        hi = lo + torch.tensor([rnd.uniform(0.4, 1.5) for _ in range(3)], device=dev)
        a, b = (lo - cam)[:, None, None] / d, (hi - cam)[:, None, None] / d
        near, ax = torch.minimum(a, b).max(dim=0)
        hit = (near < torch.maximum(a, b).amin(dim=0)) & (near > 0.05) & (near < t)
        t = torch.where(hit, near, t)
        obj = torch.where(hit, torch.full_like(obj, 6 + k), obj)
        nb = torch.zeros_like(d).scatter_(0, ax[None], -torch.sign(d.gather(0, ax[None])))
        n = torch.where(hit[None], nb, n)
    for k in range(2):  # spheres
        c = torch.tensor([rnd.uniform(1.5, 6.5), rnd.uniform(0.5, 2.5), rnd.uniform(3, 6.5)], device=dev)
        rad = rnd.uniform(0.4, 0.9)
        oc = cam - c
        bq = (d * oc[:, None, None]).sum(dim=0)
        disc = bq * bq - (oc.dot(oc) - rad * rad)
        near = -bq - disc.clamp(min=0).sqrt()
        hit = (disc > 0) & (near > 0.05) & (near < t)
        t = torch.where(hit, near, t)
        obj = torch.where(hit, torch.full_like(obj, 14 + k), obj)
        n = torch.where(hit[None], (oc[:, None, None] + near * d) / rad, n)
    p = cam[:, None, None] + t * d
    albedo = torch.tensor([[rnd.uniform(0.1, 0.9) for _ in range(3)] for _ in range(16)], device=dev)[obj].permute(2, 0, 1)
    edge = torch.minimum(p, room[:, None, None] - p).clamp(min=0).sort(dim=0).values[1]  # distance to the nearest corner line
    ao = 0.35 + 0.6 * (1 - torch.exp(-1.5 * edge))
    ao = (ao + torch.randn((H, W), device=dev, generator=gen) * torch.sqrt(ao * (1 - ao) / 64)).clamp(0, 1)
    light = torch.tensor([rnd.uniform(2, 6), 3.9, rnd.uniform(2, 6)], device=dev)[:, None, None] - p
    dist = light.square().sum(dim=0)
    tint = torch.tensor([rnd.uniform(0.6, 1.4) for _ in range(3)], device=dev)[:, None, None]
    clean = tint * (0.05 + 0.25 * ao + 1.5 * ((n * light).sum(dim=0) * torch.rsqrt(dist)).clamp(min=0) / (1 + dist))
    draw1 = -torch.log(torch.rand((1, H, W), device=dev, generator=gen).clamp(min=1e-6))
    noisy = clean * (0.5 * draw1 * draw1) * (0.8 + 0.4 * torch.rand((3, H, W), device=dev, generator=gen))
    guide = torch.cat([albedo, n, t[None] / 12.0, ao[None]])
    return guide.float().contiguous(), noisy.float().contiguous(), clean.float().contiguous()


def _weights(seed, outputs):
    """The network's parameters, flat in the library's order: per layer weights, then biases."""
    rng, parts = np.random.default_rng(seed), []
    for name, ci, co, k in LAYERS:
        co = outputs if name == "o1" else co
        b = math.sqrt(6.0 / (ci * k * k)) * (0.1 if name == "o1" else 1.0)
        parts += [rng.uniform(-b, b, co * ci * k * k), rng.uniform(-0.05, 0.05, co)]
    return np.concatenate(parts).astype(np.float32)


def _batch(seed, N, H, W):
    """N crops: network input [N, 11, H, W] and noise-free radiance [N, 3, H, W]."""
    xs, rs = [], []
    for k in range(N):
        g, y, c = _room(seed * 64 + k, H, W)
        xs.append(torch.cat([g, y]))
        rs.append(c)
    return torch.stack(xs), torch.stack(rs)


def _frame(case, seed):
    g, y, _ = _room(seed, case["H"], case["W"])
    q = case.get("q", 8)
    z = None
    if case.get("map"):
        z = (g + 0.05 * torch.roll(g, 3, dims=2)).contiguous()[:q].contiguous()
    gen = torch.Generator(device=_dev())
    gen.manual_seed(seed + 7)
    gout = torch.randn(y.shape, device=_dev(), generator=gen)
    return g[:q].contiguous(), y, z, gout


def _guide_grad(seed, N, outputs, H, W):
    """A loss's gradient at the enhanced guides: it varies over tens of pixels, as guides do."""
    gen = torch.Generator(device=_dev())
    gen.manual_seed(seed + 7)
    coarse = torch.randn((N, outputs, 4, 4), device=_dev(), generator=gen)
    return (1e-3 * F.interpolate(coarse, size=(H, W), mode="bilinear")).contiguous()


def _serving_sizes(case):
    """Frames per size and the output sizes: 2/3, 1 and 4/3 of the middle one."""
    H, W = case["H"], case["W"]
    return [(n, h, w) for n, h, w in ((case["n0"], H * 2 // 3, W * 2 // 3), (case["n1"], H, W),
                                      (case["n2"], H * 4 // 3, W * 4 // 3)) if n > 0]


def _serving_inputs(case, seed):
    groups = []
    for i, (n, h, w) in enumerate(_serving_sizes(case)):
        xs, zs = [], []
        for k in range(n):
            g, y, _ = _room(seed * 64 + 8 * i + k, h, w)
            xs.append(torch.cat([g, y])[:, ::2, ::2])
            zs.append(g)
        groups.append((torch.stack(xs).contiguous(), torch.stack(zs).contiguous()))
    return groups


# ---- one pass --------------------------------------------------------------------------------
def prepare(case, seed):
    from paper_2410_11625_gb300 import flnr, flnr_train, flr, serving
    kind = case["kind"]
    s = {"kind": kind}
    if kind in ("flr", "backward", "autograd"):
        s["g"], s["y"], s["z"], s["gout"] = _frame(case, seed)
        s["f"] = flr.FLR(q=case["q"], radius=case["r"], coef_radius=case["rc"], eps=EPS, pivot_ratio=TAU)
        s["f"].reserve(case["H"], case["W"])
        if kind == "autograd":
            for k in ("g", "y", "z"):
                if s[k] is not None:
                    s[k].requires_grad_(True)
    elif kind == "fast":
        g, y, _ = _room(seed, case["H"] * case["scale"], case["W"] * case["scale"])
        sc = case["scale"]
        s["g"], s["y"] = (t[:, ::sc, ::sc].contiguous() for t in (g, y))
        s["z"] = g if sc > 1 else None
        s["f"] = flr.FastFLR(q=8, factor=case["factor"], scale=sc, sigma=SIGMA, taps=TAPS, eps=EPS, pivot_ratio=TAU)
    elif kind in ("flnr_forward", "flnr_grads"):
        N, H, W = case["N"], case["H"], case["W"]
        s["net"] = flnr.FLNR(N * H * W, _weights(seed, case["outputs"]), outputs=case["outputs"])
        s["x"], _ = _batch(seed, N, H, W)
        if kind == "flnr_grads":
            s["gout"] = _guide_grad(seed, N, case["outputs"], H, W)
    elif kind == "train":
        x, ref = _batch(seed, case["N"], case["H"], case["W"])
        w = _weights(seed, case["outputs"])
        s["x"], s["ref"] = x.cpu().numpy(), ref.cpu().numpy()
        shape_only = flnr.init_weights(0, case["outputs"])
        tr = flnr_train.Trainer(shape_only, batch=case["N"], crop=case["H"], lr=LR, loss=case["loss"])
        for _ in range(3):  # a training under way: its step is captured, its moments are warm
            tr.step(s["x"], s["ref"])
        tr.net.set_state(np.concatenate([w, np.zeros_like(w), np.full_like(w, ADAM_RMS ** 2)]))
        tr.steps = ADAM_T
        s["tr"] = tr
    else:
        groups = [(x, z, torch.empty((z.shape[0], 3) + tuple(z.shape[2:]), device=z.device))
                  for x, z in _serving_inputs(case, seed)]
        w = _weights(seed, 8)
        s["b"] = serving.GuidedBatch(groups, w, factor=4, sigma=SIGMA, taps=TAPS, eps=EPS, pivot_ratio=TAU)
        s["out"] = [o for _, _, o in groups]
        s["done"] = torch.cuda.Event()
    return s


def run(s):
    from paper_2410_11625_gb300 import flr
    kind = s["kind"]
    if kind == "flr":
        return s["f"].denoise(s["g"], s["y"], map_guide=s["z"])
    if kind == "backward":
        return s["f"].backward(s["g"], s["y"], s["gout"], map_guide=s["z"])
    if kind == "autograd":
        leaves = [t for t in (s["g"], s["y"], s["z"]) if t is not None]
        out = flr.flr_autograd(s["f"], s["g"], s["y"], s["z"])
        return [out.detach()] + list(torch.autograd.grad(out, leaves, s["gout"]))
    if kind == "fast":
        return s["f"].denoise(s["g"], s["y"], map_guide=s["z"])
    if kind == "flnr_forward":
        return s["net"].forward(s["x"])
    if kind == "flnr_grads":
        guides = s["net"].forward(s["x"])
        s["net"].zero_grads(s["x"])
        s["net"].backward(s["gout"])
        return {"guides": guides, "grads": s["net"].grads()}
    if kind == "train":
        loss = s["tr"].step(s["x"], s["ref"])
        return {"loss": loss, "denoised": s["tr"].out, "weights": s["tr"].net.get_weights()}
    s["b"].run()
    s["done"].record(s["b"].stream)
    torch.cuda.current_stream().wait_event(s["done"])
    return s["out"]


# ---- what a pass cannot do without --------------------------------------------------------------
def _flr_flops(q, rc):
    """Per pixel: products, window sums, centring, Cholesky, triangular solves, bias, average, apply."""
    prod = q * (q + 1) // 2 + 3 * q
    f = prod + 4 * (prod + q + 3) + 2 * q + 3 + 2 * prod
    f += 2 * (q * (q - 1) // 2 + sum((q - 1 - j) * j for j in range(q))) + q * (q - 1) // 2 + 2 * q
    return f + 6 * q * q + 6 * q + (12 * (q + 1) if rc > 0 else 0) + 6 * (q + 1)


def _net_flops(N, H, W, outputs):
    res = {"e1b": 4, "e2a": 4, "e2b": 16, "d1a": 4, "d1b": 4}
    return 2 * N * H * W * sum(ci * (outputs if n == "o1" else co) * k * k / res.get(n, 1) for n, ci, co, k in LAYERS)


def _fast_flops(px_in, px_out, factor):
    return px_in * (60 + 71) + px_in / factor ** 2 * (71 * 4 * (2 * TAPS + 1) + 700) + px_out * (27 * 4 + 54)


def work(case):
    kind, H, W = case["kind"], case["H"], case["W"]
    px, q = H * W, case.get("q", 8)
    if kind == "flr":
        return {"bytes": 4 * px * (q + 6 + (q if case["map"] else 0)), "flops": px * _flr_flops(q, case["rc"])}
    if kind in ("backward", "autograd"):
        nz = q if case["map"] else 0
        b = 4 * px * (2 * (q + 3 + nz) + 3)  # inputs, the output's gradient; the gradients
        f = 3 * px * _flr_flops(q, case["rc"])
        return {"bytes": b + (12 * px if kind == "autograd" else 0), "flops": f}
    if kind == "fast":
        pxo = px * case["scale"] ** 2
        b = 4 * (px * 11 + pxo * 3 + (8 * pxo if case["scale"] > 1 else 0))
        return {"bytes": b, "flops": _fast_flops(px, pxo, case["factor"])}
    if kind == "serving":
        b = f = 0
        for n, h, w in _serving_sizes(case):
            b += 4 * n * h * w * (11 / 4 + 8 + 3)
            f += _net_flops(n, h // 2, w // 2, 8) + n * _fast_flops(h * w / 4, h * w, 4)
        return {"bytes": b, "flops": f}
    N, o = case["N"], case["outputs"]
    fwd = _net_flops(N, H, W, o)
    if kind == "flnr_forward":
        return {"bytes": 4 * N * px * (11 + o), "flops": fwd}
    params = 4 * _weights(0, o).size
    if kind == "flnr_grads":
        return {"bytes": 4 * N * px * (11 + 2 * o) + 2 * params, "flops": 3 * fwd}
    return {"bytes": 4 * N * px * (11 + 3 + 3) + 7 * params, "flops": 3 * fwd + 4 * N * px * _flr_flops(8, 8)}


# ---- float64 results in plain PyTorch -------------------------------------------------------------
def _box(t, r):
    """Sums over the window of radius r, clipped to the image, along the last two dimensions."""
    for dim in (-1, -2):
        n = t.shape[dim]
        c = torch.cat([torch.zeros_like(t.narrow(dim, 0, 1)), torch.cumsum(t, dim)], dim)
        i = torch.arange(n, device=t.device)
        t = c.index_select(dim, (i + r + 1).clamp(max=n)) - c.index_select(dim, (i - r).clamp(min=0))
    return t


def _models(mean, q):
    """Ridge models from window means: mean(name) of 'x', i / 'y', c / 'xx', i, j / 'xy', i, c.
    Returns a[i][c] and b[c]; Cholesky plane by plane."""
    mu = [mean("x", i) for i in range(q)]
    my = [mean("y", c) for c in range(3)]
    L, inv, z = {}, [], {}
    for j in range(q):
        for i in range(j, q):
            m = mean("xx", j, i) - mu[i] * mu[j] + (EPS if i == j else 0.0)
            for k in range(j):
                m = m - L[i, k] * L[j, k]
            if i == j:
                inv.append(m.rsqrt())
            else:
                L[i, j] = m * inv[j]
        for c in range(3):
            d = mean("xy", j, c) - mu[j] * my[c]
            for k in range(j):
                d = d - L[j, k] * z[k, c]
            z[j, c] = d * inv[j]
    a = {}
    for i in reversed(range(q)):
        for c in range(3):
            s = z[i, c]
            for k in range(i + 1, q):
                s = s - L[k, i] * a[k, c]
            a[i, c] = s * inv[i]
    b = [my[c] - sum(a[i, c] * mu[i] for i in range(q)) for c in range(3)]
    return a, b


def _flr64(g, y, z, r, rc):
    q = g.shape[0]
    sx = g.detach().mean(dim=(1, 2), keepdim=True)
    x, zz = g - sx, (g if z is None else z) - sx
    n = _box(torch.ones_like(y[:1]), r)[0]

    def mean(what, i, j=0):
        t = {"x": lambda: x[i], "y": lambda: y[i], "xx": lambda: x[i] * x[j], "xy": lambda: x[i] * y[j]}[what]()
        return _box(t, r) / n
    a, b = _models(mean, q)
    m = _box(torch.ones_like(y[:1]), rc)[0]
    avg = (lambda t: _box(t, rc) / m) if rc > 0 else (lambda t: t)
    return torch.stack([avg(b[c]) + sum(avg(a[i, c]) * zz[i] for i in range(q)) for c in range(3)])


def _fast64(g, y, z, factor, scale):
    q, H, W = g.shape[0], g.shape[1], g.shape[2]
    sx = g.mean(dim=(1, 2), keepdim=True)
    x, zz = g - sx, (g if z is None else z) - sx
    Hb, Wb = -(-H // factor), -(-W // factor)
    k = torch.arange(-TAPS, TAPS + 1, device=g.device, dtype=torch.float64)
    k = torch.exp(-k * k / (2 * SIGMA * SIGMA))

    def blocks(t):
        t = F.pad(t, (0, Wb * factor - W, 0, Hb * factor - H)).reshape(Hb, factor, Wb, factor).sum(dim=(1, 3))
        t = F.conv2d(t[None, None], k[None, None, None], padding=(0, TAPS))
        return F.conv2d(t, k[None, None, :, None], padding=(TAPS, 0))[0, 0]
    n = blocks(torch.ones_like(y[0]))

    def mean(what, i, j=0):
        t = {"x": lambda: x[i], "y": lambda: y[i], "xx": lambda: x[i] * x[j], "xy": lambda: x[i] * y[j]}[what]()
        return blocks(t) / n
    a, b = _models(mean, q)

    def axis(size, nb):
        c = ((torch.arange(size, device=g.device, dtype=torch.float64) + 0.5) / (factor * scale) - 0.5).clamp(0, nb - 1)
        lo = c.floor().long().clamp(max=max(nb - 2, 0))
        return lo, (lo + 1).clamp(max=nb - 1), c - lo
    y0, y1, fy = axis(H * scale, Hb)
    x0, x1, fx = axis(W * scale, Wb)

    def lerp(t):
        t = t[y0] + (t[y1] - t[y0]) * fy[:, None]
        return t[:, x0] + (t[:, x1] - t[:, x0]) * fx
    return torch.stack([lerp(b[c]) + sum(lerp(a[i, c]) * zz[i] for i in range(q)) for c in range(3)])


def _params64(flat, outputs):
    out, at = {}, 0
    for name, ci, co, k in LAYERS:
        co = outputs if name == "o1" else co
        for part, shape in ((".w", (co, ci, k, k)), (".b", (co,))):
            n = int(np.prod(shape))
            out[name + part] = torch.from_numpy(flat[at:at + n].astype(np.float64)).reshape(shape).to(_dev())
            at += n
    return out


def _net64(x, p):
    def conv(t, name, stride=1):
        w = p[name + ".w"]
        return F.conv2d(t, w, p[name + ".b"], stride=stride, padding=w.shape[-1] // 2)

    def up(t):
        return t.repeat_interleave(2, dim=2).repeat_interleave(2, dim=3)
    h = torch.cat([x[:, :8], torch.log1p(x[:, 8:].clamp(min=0))], dim=1)
    f0 = conv(conv(h, "in0").relu(), "in1").relu()
    f1 = conv(conv(f0, "e1a").relu(), "e1b", 2).relu()
    f2 = conv(conv(f1, "e2a").relu(), "e2b", 2).relu()
    d1 = conv(conv(torch.cat([up(f2), f1], dim=1), "d1a").relu(), "d1b").relu()
    d0 = conv(conv(torch.cat([up(d1), f0], dim=1), "d0a").relu(), "d0b").relu()
    return torch.sigmoid(conv(conv(d0, "o0").relu(), "o1"))


def exact(case, seed):
    kind = case["kind"]
    if kind in ("flr", "backward", "autograd"):
        g, y, z, gout = (None if t is None else t.double() for t in _frame(case, seed))
        if kind == "flr":
            return _flr64(g, y, z, case["r"], case["rc"])
        leaves = [t.requires_grad_(True) for t in (g, y, z) if t is not None]
        out = _flr64(g, y, z, case["r"], case["rc"])
        grads = torch.autograd.grad(out, leaves, gout)
        if kind == "backward":
            return dict(zip(("guide", "radiance"), grads))
        return [out.detach()] + list(grads)
    if kind == "fast":
        sc = case["scale"]
        g, y, _ = _room(seed, case["H"] * sc, case["W"] * sc)
        lo = [t[:, ::sc, ::sc].double() for t in (g, y)]
        return _fast64(lo[0], lo[1], g.double() if sc > 1 else None, case["factor"], sc)
    if kind == "serving":
        p = _params64(_weights(seed, 8), 8)
        out = []
        for x, z in _serving_inputs(case, seed):
            x = x.double()
            out.append(torch.stack([_fast64(_net64(x[k:k + 1], p)[0], x[k, 8:], z[k].double(), 4, 2)
                                    for k in range(x.shape[0])]))
        return out
    N, H, W, o = case["N"], case["H"], case["W"], case["outputs"]
    flat = _weights(seed, o)
    x, ref = _batch(seed, N, H, W)
    x, ref = x.double(), ref.double()
    p = _params64(flat, o)
    if kind == "flnr_forward":
        return _net64(x, p)
    for t in p.values():
        t.requires_grad_(True)
    if kind == "flnr_grads":
        guides = _net64(x, p)
        grads = torch.autograd.grad(guides, list(p.values()), _guide_grad(seed, N, o, H, W).double())
        return {"guides": guides.detach(), "grads": torch.cat([t.reshape(-1) for t in grads])}
    guides = _net64(x, p)
    den = torch.stack([_flr64(guides[k, :8], x[k, 8:], guides[k, 8:] if o == 16 else None, 8, 8) for k in range(N)])
    err = (den - ref).abs()
    loss = (err if case["loss"] == "l1" else err / (den.abs() + ref.abs() + 0.01)).mean()
    grad = torch.cat([t.reshape(-1) for t in torch.autograd.grad(loss, list(p.values()))])
    m, v = (1 - BETA1) * grad, BETA2 * ADAM_RMS ** 2 + (1 - BETA2) * grad * grad
    step = LR * (m / (1 - BETA1 ** (ADAM_T + 1))) / ((v / (1 - BETA2 ** (ADAM_T + 1))).sqrt() + ADAM_EPS)
    w = torch.from_numpy(flat.astype(np.float64)).to(grad.device) - step
    return {"loss": loss.detach().reshape(1), "denoised": den.detach(), "weights": w}
