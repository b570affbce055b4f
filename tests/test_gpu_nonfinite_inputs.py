"""The classifier on particles so far out that its inputs overflow BF16.

Such a particle lies outside every mesh; its window is infinite in one channel
and its start is of no use, but its logits have to be those of the network: a
logit is NaN or infinite where the sums that lead to it are, and finite
elsewhere. The reference evaluates the layers in FP64 from the library's own
inputs, rounding operands to BF16 where the kernels do, and leaves out what lies
in the zero padding. Bar: the kind of every logit (finite, +-Inf, NaN), and the
finite ones to 3e-2 of their row's size, the BF16 rounding of six layers
(2^-9 a value and layer, sqrt(6) 2^-9 = 5e-3 in a row's norm, six times that
allowed). Particles of the same call that lie in the mesh have finite logits,
also those that share a tile with one that has not."""

import numpy as np
import pytest

from workloads import make_case
from workloads.weights import classifier_layer_shapes, init_classifier

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2412_18379_gb300 as cs
    from paper_2412_18379_gb300 import build
    build.build()
    c = cs.Context(0)
    yield c
    c.close()


def _bf16(a):
    """Rounded to BF16, overflow to infinity, as FP64."""
    import torch
    return torch.from_numpy(np.asarray(a, np.float64)).to(torch.float32).to(torch.bfloat16) \
        .to(torch.float64).numpy()


def _relu(z):
    return np.where(z > 0, z, 0.0)      # a NaN gives 0, as fmaxf


def _conv(x, W, b, dim):
    """Zero-padded 3^dim convolution of x [n, C, S..]; products with the padding
    are left out of the sums."""
    n, S = x.shape[0], x.shape[2]
    out = np.zeros((n, W.shape[0]) + (S,) * dim) + b.reshape((1, -1) + (1,) * dim)
    for t in range(3 ** dim):
        o = [t // 3 ** k % 3 - 1 for k in range(dim)][::-1]       # slowest axis first
        dst = tuple(slice(max(0, -d), S - max(0, d)) for d in o)
        src = tuple(slice(max(0, d), S + min(0, d)) for d in o)
        with np.errstate(invalid="ignore"):
            out[(slice(None), slice(None)) + dst] += np.einsum(
                "oc,nc...->no...", W[:, :, t], x[(slice(None), slice(None)) + src])
    return out


def _logits(params, win, off, dim):
    p, o = [], 0
    for ws, bs in classifier_layer_shapes(dim):
        for s in (ws, bs):
            k = int(np.prod(s))
            p.append(params[o:o + k].reshape(s).astype(np.float64))
            o += k
    W = [_bf16(w) for w in p[0::2]]
    b = p[1::2]
    with np.errstate(invalid="ignore", over="ignore"):
        y = _bf16(_relu(_conv(_bf16(win), W[0], b[0], dim)))
        y = _relu(_conv(y, W[1], b[1], dim))
        S = y.shape[2]
        h = 2 * (S // 2)
        y = y[(slice(None), slice(None)) + (slice(0, h),) * dim]
        y = y.reshape(y.shape[:2] + sum(((h // 2, 2) for _ in range(dim)), ()))
        y = y.mean(axis=tuple(3 + 2 * k for k in range(dim))).reshape(y.shape[0], -1)
        r = _bf16(off)
        for l in (2, 3):
            r = _bf16(_relu(r @ W[l].T + b[l]))
        u = _bf16(_relu(np.concatenate([_bf16(y), r], axis=1) @ W[4].T + b[4]))
        return u @ W[5].T + b[5]


def _kinds(g):
    return np.where(np.isnan(g), 3, np.where(g == np.inf, 1, np.where(g == -np.inf, 2, 0)))


@pytest.mark.parametrize("dim,n", [(2, 40), (2, 2300), (2, 9), (3, 40)])
def test_logits_of_overflowing_windows(ctx, dim, n):
    """Few particles take a tile each, 15 per SM and more five in 2-D; fewer than 16
    rows have their own fully connected layers."""
    c = make_case("tg2d", n_side=41) if dim == 2 else make_case("abc3d", n_side=9)
    rng = np.random.default_rng(n)
    xp = rng.random((n, dim))
    far = np.arange(0, min(n, 40), 3)
    for i in far:
        xp[i, i % dim] = (1.0, 3.0, -1.0, -3.0)[i % 4] * 1e38
    for seed in range(4):
        params = init_classifier(dim, seed)
        ctx.load_classifier(dim, params)
        mesh = ctx.upload_mesh(c.xyz, c.conn)
        import torch
        x = torch.from_numpy(xp).cuda()
        win, off = ctx.classifier_features(mesh, x)
        got = ctx.classifier_forward(mesh, x).cpu().numpy().astype(np.float64)
        mesh.release()
        rows = np.arange(min(n, 45))
        S = 9 if dim == 2 else 7
        want = _logits(params, win.cpu().numpy()[rows].reshape((-1, dim) + (S,) * dim),
                       off.cpu().numpy()[rows], dim)
        near = np.setdiff1d(np.arange(n), far)
        assert np.isfinite(got[near]).all()
        assert np.array_equal(_kinds(got[rows]), _kinds(want)), seed
        fin = np.isfinite(want).all(axis=1)
        err = np.linalg.norm(got[rows][fin] - want[fin], axis=1)
        assert np.all(err <= 3e-2 * np.linalg.norm(want[fin], axis=1))
