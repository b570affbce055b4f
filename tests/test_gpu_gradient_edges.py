"""Gradients of the fused training kernels at the edges of their tiles, against
a plain evaluation in FP64 that rounds to BF16 where the kernels do.

Both sides hold the same BF16 operands but for values whose FP32 and FP64 sums
fall on different sides of a rounding boundary. A sum of K terms errs by about
sqrt(K) 2^-24 of its terms' size, so for K = 864 one value in
2^-9 / (30 2^-24) = 1100 is one BF16 step (2^-8 of it) off: in norm
2^-8 / sqrt(1100) = 1.2e-4 a layer, sqrt(12) of that over the six layers'
forward and backward values, 4e-4, and as much again for the ReLUs that open or
close with such a value. Allowed: 3e-3 of each layer's gradient in norm. A row
left out, doubled or put in another's place in a batch of B shows at about
1 / sqrt(B) >= 2.5e-2, a tap or a channel in another's place at its full size.
The sizes leave one input over, fill a tile, or add a tile per SM (152)."""

import numpy as np
import pytest

from oracle import cnn
from workloads import make_case
from workloads.weights import classifier_layer_shapes, init_classifier, init_weights, layer_shapes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2412_18379_gb300 as cs
    from paper_2412_18379_gb300 import build
    build.build()
    c = cs.Context(0)
    yield c
    c.close()


def _bf(x):
    import torch
    return x.to(torch.float32).to(torch.bfloat16).to(torch.float64)


def _unpack(flat, shapes):
    import torch
    p, o = [], 0
    for ws, bs in shapes:
        for s in (ws, bs):
            n = int(np.prod(s))
            p.append(torch.from_numpy(flat[o:o + n].astype(np.float64)).reshape(s).cuda())
            o += n
    return p[0::2], p[1::2]


def _conv(x, W, b, dim, pad):
    import torch
    w = _bf(W).reshape(W.shape[:2] + (3,) * dim)
    f = torch.nn.functional.conv2d if dim == 2 else torch.nn.functional.conv3d
    return f(x, w, b, padding=pad)


def _conv_back(x, W, dz, dim, pad):
    """(weight gradient, input gradient) from BF16 dz."""
    import torch
    w = _bf(W).reshape(W.shape[:2] + (3,) * dim)
    g = torch.nn.grad
    wg, xg = (g.conv2d_weight, g.conv2d_input) if dim == 2 else (g.conv3d_weight, g.conv3d_input)
    d = _bf(dz)
    return wg(x, w.shape, d, padding=pad).reshape(W.shape), xg(x.shape, w, d, padding=pad)


def _regressor(flat, win, tgt, dim):
    shapes = layer_shapes(dim)
    W, b = _unpack(flat, shapes)
    n = len(shapes) - 2
    x = [_bf(win.double())]
    for l in range(n):
        x.append(_bf(_conv(x[l], W[l], b[l], dim, 0).clamp(min=0)))
    h = x[n].flatten(1)
    a5 = _bf((h @ _bf(W[n]).T + b[n]).clamp(min=0))
    e = a5 @ _bf(W[n + 1]).T + b[n + 1] - tgt.double()
    gout = 2 * e / e.numel()
    dW, db = [None] * (n + 2), [None] * (n + 2)
    dW[n + 1], db[n + 1] = _bf(gout).T @ a5, gout.sum(0)
    da = (_bf(gout) @ _bf(W[n + 1])) * (a5 > 0)
    dW[n], db[n] = _bf(da).T @ h, da.sum(0)
    dz = ((_bf(da) @ _bf(W[n])) * (h > 0)).reshape(x[n].shape)
    for l in range(n - 1, -1, -1):
        db[l] = dz.transpose(0, 1).flatten(1).sum(1)
        dW[l], dx = _conv_back(x[l], W[l], dz, dim, 0)
        dz = dx * (x[l] > 0)
    return dW, db


def _classifier(flat, win, off, lab, dim):
    import torch
    W, b = _unpack(flat, classifier_layer_shapes(dim))
    S = 9 if dim == 2 else 7
    x0 = _bf(win.double().reshape((-1, dim) + (S,) * dim))
    x1 = _bf(_conv(x0, W[0], b[0], dim, 1).clamp(min=0))
    z2 = _conv(x1, W[1], b[1], dim, 1)
    pool = torch.nn.functional.avg_pool2d if dim == 2 else torch.nn.functional.avg_pool3d
    z2 = z2.requires_grad_(True)
    pooled = pool(z2.clamp(min=0), 2)
    o = _bf(off.double())
    r1 = _bf((o @ _bf(W[2]).T + b[2]).clamp(min=0))
    h2 = _bf((r1 @ _bf(W[3]).T + b[3]).clamp(min=0))
    cat = torch.cat([_bf(pooled.detach().flatten(1)), h2], 1)
    ru = _bf((cat @ _bf(W[4]).T + b[4]).clamp(min=0))
    H = ru @ _bf(W[5]).T + b[5]
    valid = (lab >= 0) & (lab < H.shape[1])
    n = int(valid.sum())
    p = torch.softmax(H, 1)
    t = torch.zeros_like(H)
    t[torch.arange(len(lab), device="cuda")[valid], lab[valid].long()] = 1
    gH = (p - t) * valid[:, None] / max(n, 1)
    dW, db = [None] * 6, [None] * 6
    dW[5], db[5] = _bf(gH).T @ ru, gH.sum(0)
    gu = (_bf(gH) @ _bf(W[5])) * (ru > 0)
    dW[4], db[4] = _bf(gu).T @ cat, gu.sum(0)
    gc = _bf(gu) @ _bf(W[4])
    npool = pooled[0].numel()
    g2 = gc[:, npool:] * (h2 > 0)
    dW[3], db[3] = _bf(g2).T @ r1, g2.sum(0)
    g1 = (_bf(g2) @ _bf(W[3])) * (r1 > 0)
    dW[2], db[2] = _bf(g1).T @ o, g1.sum(0)
    pooled.backward(gc[:, :npool].reshape(pooled.shape))
    dz = z2.grad
    for l, x in ((1, x1), (0, x0)):
        db[l] = dz.transpose(0, 1).flatten(1).sum(1)
        dW[l], dx = _conv_back(x, W[l], dz, dim, 1)
        dz = dx * (x > 0)
    return dW, db


def _check(flat, dW, db, shapes):
    o = 0
    for l, (ws, bs) in enumerate(shapes):
        for want, s in ((dW[l], ws), (db[l], bs)):
            n = int(np.prod(s))
            got = flat[o:o + n].double().reshape(tuple(s))
            rel = float((got - want).norm() / want.norm())
            assert rel <= 3e-3, (l, "W" if want is dW[l] else "b", rel)
            o += n


@pytest.mark.parametrize("dim,B", [(2, 15), (2, 16), (2, 17), (2, 153), (2, 609), (2, 1521),
                                   (3, 15), (3, 16), (3, 17), (3, 153), (3, 609)])
def test_regressor(ctx, dim, B):
    import torch
    flat = init_weights(dim, 29)
    ctx.load_predictor(dim, flat)
    gen = torch.Generator(device="cuda").manual_seed(B)
    S = cnn.patch_size(dim)
    win = torch.randn((B, dim) + (S,) * dim, generator=gen, device="cuda")
    tgt = torch.randn((B, dim), generator=gen, device="cuda")
    g, _ = ctx.predictor_grad(dim, win, tgt)
    ctx.device_status()
    dW, db = _regressor(flat, win, tgt, dim)
    _check(g, dW, db, layer_shapes(dim))


@pytest.mark.parametrize("dim,B", [(2, 15), (2, 16), (2, 17), (2, 129), (2, 153), (2, 609),
                                   (3, 15), (3, 17)])
def test_classifier(ctx, dim, B):
    import torch
    c = make_case("tg2d", n_side=41) if dim == 2 else make_case("abc3d", n_side=9)
    flat = init_classifier(dim, 31)
    ctx.load_classifier(dim, flat)
    mesh = ctx.upload_mesh(c.xyz, c.conn)
    gen = torch.Generator(device="cuda").manual_seed(B)
    xp = torch.rand((B, dim), dtype=torch.float64, generator=gen, device="cuda")
    lab = torch.randint(-1, 81 if dim == 2 else 343, (B,), dtype=torch.int32, generator=gen,
                        device="cuda")
    win, off = ctx.classifier_features(mesh, xp)
    g, _ = ctx.classifier_grad(mesh, xp, lab)
    dW, db = _classifier(flat, win, off, lab, dim)
    _check(g, dW, db, classifier_layer_shapes(dim))
    mesh.release()


@pytest.mark.parametrize("dim,n", [(2, 8192 + 15), (2, 8192 + 16), (2, 2 * 8192 + 1), (3, 8200)])
def test_forward_chunks(ctx, dim, n):
    """Windows are taken 8192 at a time; the last chunk, of whichever path takes
    so few, has the outputs of a call of its own."""
    import torch
    ctx.load_predictor(dim, init_weights(dim, 5))
    gen = torch.Generator(device="cuda").manual_seed(n)
    S = cnn.patch_size(dim)
    win = torch.randn((n, dim) + (S,) * dim, generator=gen, device="cuda")
    out = ctx.predictor_forward(dim, win)
    for a in range(0, n, 8192):
        own = ctx.predictor_forward(dim, win[a:a + 8192].contiguous())
        assert torch.equal(out[a:a + 8192], own)
