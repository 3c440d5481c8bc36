"""The training kernels in the forms that large batches run (tall tiles of the
convolutions, several tiles and sums per block of the weight gradient), against
the same network in FP64 through torch.

Rounding of the weight gradients: networks of identity kernels, positive images
of few bits and targets at a few bits' distance from the network's output, so
that every activation and every gradient of one is exact in FP32 and a weight
gradient's only error is that of its own sum. A sum of n terms that ends every
F terms has n / F chains whose partial sums grow as sqrt(j): an RMS error of
c sqrt((F + 1) / 2) units of 2^-24 over the root of the sum of its squared
terms, where c, the RMS rounding error of a number in units of its own 2^-24,
is at most 1 / sqrt(3). The bound is that of sums of 8 pixels added up by 304
blocks, F = 8 + n / 2432, and one rounding of the result. The terms of a sum
have to be independent for this: the network that stops at the first level
serves for that level's layers, the other one for the layers below."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _shapes(ci, co):
    return [(ci, 16), (16, 16), (16, 32), (32, 32), (32, 32), (32, 32), (64, 32), (48, 16), (16, co)]


def _forward(par, x, shapes):
    """The network in par's precision: output, every layer's input and result."""
    import torch
    f = torch.nn.functional
    at, layers = 0, []
    for ci, co in shapes:
        w = par[at:at + 9 * ci * co].view(3, 3, ci, co).permute(3, 2, 0, 1)
        layers.append((w, par[at + 9 * ci * co:at + 9 * ci * co + co]))
        at += 9 * ci * co + co
    ins, pre = [], []

    def layer(k, v):
        ins.append(v)
        pre.append(f.conv2d(v, layers[k][0], layers[k][1], padding=1))
        pre[-1].retain_grad()
        return pre[-1] if k == 8 else pre[-1].relu()

    def up(v):
        return f.interpolate(v, scale_factor=2, mode="bilinear", align_corners=False)

    s1 = layer(1, layer(0, x.permute(0, 3, 1, 2)))
    s2 = layer(3, layer(2, f.avg_pool2d(s1, 2)))
    c2 = layer(5, layer(4, f.avg_pool2d(s2, 2)))
    d1 = layer(6, torch.cat([up(c2), s2], 1))
    e1 = layer(7, torch.cat([up(d1), s1], 1))
    return layer(8, e1).permute(0, 2, 3, 1), ins, pre


def _identity_params(deep):
    """Every layer passes its channels on (the decoder's also the skipped ones);
    without `deep` the levels below the first pass nothing."""
    out = []
    for k, (ci, co) in enumerate(_shapes(16, 2)):
        w = np.zeros((3, 3, ci, co), np.float32)
        if k in (0, 1):
            w[1, 1] = np.eye(16)
        elif k == 2 and deep:
            w[1, 1] = np.concatenate([np.eye(16)] * 2, 1)
        elif k in (3, 4, 5) and deep:
            w[1, 1] = np.eye(32)
        elif k == 6 and deep:
            w[1, 1] = np.concatenate([np.eye(32)] * 2, 0)
        elif k == 7:
            w[1, 1] = np.concatenate([np.eye(32)[:, :16] * deep, np.eye(16)], 0)
        elif k == 8:
            w[1, 1] = np.eye(16)[:, :2]
        out += [w.ravel(), np.zeros(co, np.float32)]
    return np.concatenate(out)


@pytest.mark.parametrize("deep", [0, 1])
@pytest.mark.parametrize("n,h,w", [(1, 64, 64), (2, 128, 128), (1, 260, 292), (8, 256, 256)])
def test_weight_gradient_rounding(lib, n, h, w, deep):
    import torch
    gk = lib
    shapes = _shapes(16, 2)
    gen = torch.Generator("cuda").manual_seed(11)
    q = 2 ** (8 if deep else 11)
    x = torch.randint(1, q + 1, (n, h, w, 16), generator=gen, device="cuda").double() / q
    noise = torch.randint(-2 ** 11, 2 ** 11 + 1, (n, h, w, 2), generator=gen, device="cuda").double() / 2 ** 11
    par = torch.tensor(_identity_params(deep), device="cuda").double().requires_grad_(True)
    y, ins, pre = _forward(par, x, shapes)
    t = y.detach() + noise
    assert torch.equal(t.float().double(), t)
    (y - t).square().sum().div(n).backward()

    u = gk.gkb_unet_create(16, 16, 32, 2, 1, torch.cuda.current_stream().cuda_stream)
    try:
        gk.gkb_unet_set_params(u, par.detach().float())
        g = torch.empty(par.numel(), dtype=torch.float32, device="cuda")
        out = torch.empty(n, h, w, 2, dtype=torch.float32, device="cuda")
        gk.gkb_unet_forward(u, x.float(), n, h, w, out, 0)
        assert torch.equal(out.double(), y.detach())
        gk.gkb_unet_loss_grad(u, x.float(), t.float().contiguous(), n, h, w, g)
    finally:
        gk.gkb_unet_destroy(u)
    at = 0
    with torch.no_grad():
        for k, (ci, co) in enumerate(shapes):
            sq = 0
            for i in range(n):
                a = torch.nn.functional.unfold(ins[k][i:i + 1].square(), 3, padding=1)[0]
                sq = sq + a @ pre[k].grad[i].reshape(co, -1).square().T
            sq = sq.view(ci, 9, co).permute(1, 0, 2).reshape(-1)
            sq = torch.cat([sq, pre[k].grad.square().sum((0, 2, 3))])
            err = (g[at:at + sq.numel()].double() - par.grad[at:at + sq.numel()]) * 2 ** 24
            on = sq > 0
            assert bool((err[~on] == 0).all())
            at += sq.numel()
            if not bool(on.any()):
                continue
            if deep != (k in (2, 3, 4, 5, 6)):
                continue
            px = n * h * w // (1 if k in (0, 1, 7, 8) else 16 if k in (4, 5) else 4)
            # the coarser levels' gradients are means over neighbours: a
            # correlation of 0.3 and a rounding of their own
            f = (8 + px / 2432 + 1) / 2
            bound = math.sqrt(f + 1) / math.sqrt(3) if k in (0, 1, 7, 8) else 1.75 * math.sqrt(f + 2) / math.sqrt(3)
            rms = float((err[on] / sq[on].sqrt()).square().mean().sqrt())
            print("layer %d: %.2f of %.2f" % (k, rms, bound))
            assert rms <= bound, (k, rms, bound)


@pytest.mark.parametrize("n,h,w,ci,co,skew", [(4, 260, 292, 3, 2, 0), (2, 332, 212, 4, 3, 1), (9, 148, 68, 13, 1, 0),
                                              (1, 512, 260, 5, 2, 0), (3, 20, 1028, 16, 3, 0)])
def test_large_training_step(lib, n, h, w, ci, co, skew):
    """Loss and gradients at sizes that take the tall tiles, ragged at every
    side, with 1 to 16 inputs (`skew`: at an address that allows no vector
    loads). Half of the channels are kept positive and half negative by their
    biases, ten deviations from zero, so that no rounding error decides a ReLU.
    FP32 sums of at most 576 terms through nine layers and back keep 1e-4 of a
    layer's norm; a pixel column or a tap left out would change 1e-2."""
    import torch
    gk = lib
    shapes = _shapes(ci, co)
    gen = torch.Generator("cuda").manual_seed(5)
    parts = []
    for k, (a, b) in enumerate(shapes):
        parts.append(torch.randn(9 * a * b, generator=gen, device="cuda") * 0.1 / math.sqrt(9 * a))
        sign = torch.ones(b, device="cuda")
        if k < 8:
            sign[1::2] = -1
        parts.append(sign * 3)
    p = torch.cat(parts)
    par = p.double().requires_grad_(True)
    x = torch.randn(n, h, w, ci, generator=gen, device="cuda")
    t = torch.randn(n, h, w, co, generator=gen, device="cuda")
    loss = 0.0
    for i in range(n):
        y, _, _ = _forward(par, x[i:i + 1].double(), shapes)
        part = (y - t[i:i + 1].double()).square().sum() / n
        part.backward()
        loss += float(part.detach())
    buf = torch.zeros(x.numel() + 4, device="cuda")
    xs = buf[skew:skew + x.numel()]
    xs.copy_(x.reshape(-1))
    u = gk.gkb_unet_create(ci, 16, 32, co, 1, torch.cuda.current_stream().cuda_stream)
    try:
        gk.gkb_unet_set_params(u, p)
        g = torch.empty(p.numel(), dtype=torch.float32, device="cuda")
        got = gk.gkb_unet_loss_grad(u, xs, t, n, h, w, g)
    finally:
        gk.gkb_unet_destroy(u)
    assert abs(got - loss) <= 1e-5 * loss
    at = 0
    for a, b in shapes:
        m = 9 * a * b + b
        ref = par.grad[at:at + m]
        assert float((g[at:at + m].double() - ref).norm()) <= 1e-4 * float(ref.norm()), (a, b)
        at += m
