"""The classifier's logits of fewer than 16 rows.

Such a batch, or the last chunk of a larger one, runs its fully connected
layers on the CUDA cores, in FP32 fused multiply-adds over k in increasing
order; the tensor cores, which take the larger ones, add in another order. The
parameters here make the last layer's input known: with zero weights before it,
each hidden value is BF16(ReLU(b4)) whatever the particle. The logits then are

  H[n] = fma(r[511], w[n][511], .. fma(r[1], w[n][1], fma(r[0], w[n][0], 0))) + b5[n]

with r and w of 8 significant bits. The reference adds each exact product in
FP64 and rounds to FP32: the fused multiply-add's bits unless the FP64 sum falls
within 2^-29 of a rounding boundary without being exact, so the comparison is of
bits."""

import numpy as np
import pytest

from workloads import make_case
from workloads.weights import classifier_layer_shapes

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
    """FP32 values rounded to BF16 (to nearest even; finite values)."""
    b = np.ascontiguousarray(a, np.float32).view(np.uint32).astype(np.uint64)
    b = (b + 0x7fff + ((b >> 16) & 1)) & 0xffff0000
    return b.astype(np.uint32).view(np.float32)


def _params(dim):
    rng = np.random.default_rng(dim)
    shapes = classifier_layer_shapes(dim)
    p = [[np.zeros(ws, np.float32), np.zeros(bs, np.float32)] for ws, bs in shapes]
    p[4][1][:] = rng.standard_normal(shapes[4][1])
    p[5][0][:] = rng.standard_normal(shapes[5][0])
    p[5][1][:] = rng.standard_normal(shapes[5][1])
    r = _bf16(np.maximum(p[4][1], 0.0)).astype(np.float64)
    w = _bf16(p[5][0]).astype(np.float64)
    acc = np.zeros(w.shape[0], np.float32)
    for k in range(w.shape[1]):
        acc = (acc.astype(np.float64) + r[k] * w[:, k]).astype(np.float32)
    return np.concatenate([x.ravel() for l in p for x in l]), acc + p[5][1]


@pytest.mark.parametrize("dim,n,rows", [(2, 1, 1), (2, 7, 7), (2, 15, 15), (2, 32768 + 8, 8),
                                        (3, 1, 1), (3, 15, 15), (3, 16384 + 15, 15)])
def test_sums_of_few_rows_run_in_order(ctx, dim, n, rows):
    import torch
    c = make_case("tg2d", n_side=41) if dim == 2 else make_case("abc3d", n_side=9)
    params, want = _params(dim)
    ctx.load_classifier(dim, params)
    mesh = ctx.upload_mesh(c.xyz, c.conn)
    gen = torch.Generator(device="cuda").manual_seed(n)
    xp = torch.rand((n, dim), dtype=torch.float64, generator=gen, device="cuda")
    H = ctx.classifier_forward(mesh, xp).cpu().numpy()
    for row in H[-rows:]:
        assert np.array_equal(row.view(np.uint32), want.view(np.uint32))
    # the other rows: the same sum in another order of FP32 additions, each
    # within 2^-23 of its terms' magnitudes added up (512 terms, 16 to a step)
    scale = np.abs(_bf16(np.maximum(params[-want.size * 513 - 512:-want.size * 513], 0.0))) @ \
        np.abs(_bf16(params[-want.size * 513:-want.size]).reshape(want.size, 512)).T
    assert np.all(np.abs(H - want) <= 512 * 2.0 ** -23 * (scale + np.abs(want)))
    mesh.release()


@pytest.mark.parametrize("dim,chunk", [(2, 32768), (3, 16384)])
def test_a_short_last_chunk(ctx, dim, chunk):
    """Its rows have the logits of a call of their own, and a larger call after
    it finds its packed weights in place."""
    import torch
    from workloads.weights import init_classifier
    c = make_case("tg2d", n_side=41) if dim == 2 else make_case("abc3d", n_side=9)
    ctx.load_classifier(dim, init_classifier(dim, 5))
    mesh = ctx.upload_mesh(c.xyz, c.conn)
    gen = torch.Generator(device="cuda").manual_seed(dim)
    xp = torch.rand((chunk + 15, dim), dtype=torch.float64, generator=gen, device="cuda")
    own = [ctx.classifier_forward(mesh, xp[a:b].contiguous())
           for a, b in ((chunk, chunk + 15), (0, chunk))]
    H = ctx.classifier_forward(mesh, xp)
    assert torch.equal(H[chunk:], own[0]) and torch.equal(H[:chunk], own[1])
    mesh.release()
