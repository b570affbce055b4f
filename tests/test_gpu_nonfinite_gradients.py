"""Gradients where an activation or a weight of a convolution is not finite.

The backward convolutions multiply, beside the products of the sums, zeros at
positions that meet no output; zero times infinity must not leave a NaN there.
Each batch of 8 rows runs layer by layer (im2col, which has no such products);
repeated twice it takes the fused kernels. The mean gradient is the same, so
every entry has to be of the same kind: finite, +Inf, -Inf or NaN.

The networks are random but for a channel that carries the corner of the
window to the layer under test, where it overflows (its weights there are -1,
so what reads it is closed by the ReLU and the loss stays finite), or, for
weights, is the only place where the channel is positive and meets only taps
with finite weights."""

import numpy as np
import pytest

from oracle import cnn
from workloads import make_case
from workloads.weights import classifier_layer_shapes, layer_shapes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2412_18379_gb300 as cs
    from paper_2412_18379_gb300 import build
    build.build()
    c = cs.Context(0)
    yield c
    c.close()


def _random(shapes, seed):
    rng = np.random.default_rng(seed)
    return [[rng.standard_normal(ws) * np.sqrt(2.0 / np.prod(ws[1:])), np.zeros(bs)]
            for ws, bs in shapes]


def _flat(p):
    return np.concatenate([np.asarray(x, np.float32).ravel() for l in p for x in l])


def _kinds(g):
    g = np.asarray(g, np.float64)
    return np.where(np.isnan(g), 3, np.where(g == np.inf, 1, np.where(g == -np.inf, 2, 0)))


def _compare(dim, shapes, few, many):
    o = 0
    for li, (ws, bs) in enumerate(shapes):
        for what, s in (("W", ws), ("b", bs)):
            n = int(np.prod(s))
            a, b = _kinds(few[o:o + n]).reshape(s), _kinds(many[o:o + n]).reshape(s)
            assert np.array_equal(a, b), (li, what, np.argwhere(a != b)[:4])
            o += n


@pytest.mark.parametrize("dim,layer", [(2, 1), (2, 2), (2, 3), (3, 1), (3, 2)])
@pytest.mark.parametrize("kind", ["activation", "weight"])
def test_regressor(ctx, dim, layer, kind):
    import torch
    shapes = layer_shapes(dim)
    p = _random(shapes, 10 * dim + layer)
    rng = np.random.default_rng(layer)
    S = cnn.patch_size(dim)
    win = rng.standard_normal((8, dim) + (S,) * dim).astype(np.float32)
    corner = (slice(None), 0) + (0,) * dim
    for l in range(layer):                      # channel 0 carries window channel 0's corner
        p[l][0][0] = 0.0
        p[l][0][:, 0] = 0.0
        p[l][0][0, 0, 0] = 1.0
    if kind == "activation":
        win[corner] = 1e38
        p[layer - 1][0][0, 0, 0] = 10.0
        p[layer][0][:, 0] = -1.0
    else:
        win[:, 0] = -np.abs(win[:, 0])
        win[corner] = 1.0
        p[layer][0][3, 0, (3 ** dim) // 2] = -np.inf     # the centre tap: not the corner's
    ctx.load_predictor(dim, _flat(p))
    tgt = torch.from_numpy(rng.standard_normal((8, dim)).astype(np.float32)).cuda()
    win = torch.from_numpy(win).cuda()
    few, lf = ctx.predictor_grad(dim, win, tgt)
    many, lm = ctx.predictor_grad(dim, win.repeat((2,) + (1,) * (dim + 1)).contiguous(),
                                  tgt.repeat(2, 1).contiguous())
    assert np.isfinite(lf) and np.isfinite(lm)
    few, many = few.cpu().numpy(), many.cpu().numpy()
    # the infinite weights' products meet zeros of a closed ReLU alone
    assert np.isfinite(few).all() if kind == "weight" else np.isnan(few).any()
    _compare(dim, shapes, few, many)


@pytest.mark.parametrize("kind", ["activation", "weight"])
def test_classifier(ctx, kind):
    """The second convolution of the 2-D classifier. Particles at ASG cell
    centres: window channel 0 grows by about one per column, and a first weight
    between 3.4e38 / 4 and 3.4e38 / 3 makes the last column alone infinite."""
    import torch
    c = make_case("tg2d", n_side=41)
    shapes = classifier_layer_shapes(2)
    p = _random(shapes, 3)
    p[0][0][0] = 0.0
    if kind == "activation":
        p[0][0][0, 0, 4] = 9.7e37
        p[1][0][:, 0] = -1.0
    else:
        # channel 0 is positive in the last column alone, which the left taps'
        # infinite weights do not meet
        p[0][0][0, 0, 4], p[0][1][0] = 1.0, -3.5
        p[1][0][3, 0, 0] = p[1][0][3, 0, 3] = p[1][0][3, 0, 6] = -np.inf
    ctx.load_classifier(2, _flat(p))
    mesh = ctx.upload_mesh(c.xyz, c.conn)
    info = mesh.info()
    lo, hi = np.array(info["lo"][:2]), np.array(info["hi"][:2])
    g = np.array(info["asg_grid"][:2])
    cells = np.stack([g // 2 + i for i in range(-4, 4)])
    xp = torch.from_numpy(lo + (cells + 0.5) * (hi - lo) / g).cuda()
    lab = torch.arange(8, dtype=torch.int32, device="cuda") * 9
    few, _ = ctx.classifier_grad(mesh, xp, lab)
    many, _ = ctx.classifier_grad(mesh, xp.repeat(2, 1).contiguous(), lab.repeat(2).contiguous())
    few, many = few.cpu().numpy(), many.cpu().numpy()
    # the infinite weights' products meet zeros of a closed ReLU alone
    assert np.isfinite(few).all() if kind == "weight" else np.isnan(few).any()
    _compare(2, shapes, few, many)
    mesh.release()
