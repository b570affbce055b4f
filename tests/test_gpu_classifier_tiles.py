"""The classifier's tiled kernels at the edges of their row tiles.

Activations travel in tiles of 128 rows, the fused convolutions take one
particle per CTA pass, inference runs in chunks of 32768 (2-D) or 16384 (3-D)
rows, and the fusion layer splits its K below 9728 rows on a 152-SM GPU.
Each row's logits depend on that row and the number of rows of its chunk
alone, so permuting the rows of a chunk permutes the logits bit for bit. The
gradients are sums over the batch: a permutation changes only the order of
FP32 sums, sqrt(2000 * 81) 2^-24 = 2.4e-5 of the terms, allowed 2e-4 in norm.
"""

import numpy as np
import pytest

from workloads import make_case
from workloads.weights import init_classifier

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2412_18379_gb300 as cs
    from paper_2412_18379_gb300 import build
    build.build()
    c = cs.Context(0)
    yield c
    c.close()


def _mesh(ctx, dim):
    c = make_case("tg2d", n_side=41) if dim == 2 else make_case("abc3d", n_side=9)
    ctx.load_classifier(dim, init_classifier(dim, 5))
    return ctx.upload_mesh(c.xyz, c.conn)


def _points(dim, n, seed):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    xp = torch.rand((n, dim), dtype=torch.float64, generator=gen, device="cuda") * 1.1 - 0.05
    perm = torch.randperm(n, generator=gen, device="cuda")
    lab = torch.randint(-1, 81 if dim == 2 else 343, (n,), dtype=torch.int32, generator=gen,
                        device="cuda")
    return xp, lab, perm


@pytest.mark.parametrize("dim,n", [(2, 1), (2, 17), (2, 128), (2, 129), (2, 9727), (2, 9729),
                                   (2, 32768), (3, 1), (3, 129), (3, 3300), (3, 9729)])
def test_permuted_rows(ctx, dim, n):
    mesh = _mesh(ctx, dim)
    xp, _, perm = _points(dim, n, n)
    H = ctx.classifier_forward(mesh, xp)
    Hp = ctx.classifier_forward(mesh, xp[perm].contiguous())
    assert bool(H.isfinite().all())
    assert np.array_equal(Hp.cpu().numpy().view(np.uint32), H[perm].cpu().numpy().view(np.uint32))
    mesh.release()


@pytest.mark.parametrize("dim,n,chunk", [(2, 32768 + 9729, 32768), (3, 16384 + 9729, 16384)])
def test_chunks(ctx, dim, n, chunk):
    """A chunk's rows have the logits of a call of their own."""
    mesh = _mesh(ctx, dim)
    xp, _, _ = _points(dim, n, 3)
    H = ctx.classifier_forward(mesh, xp).cpu().numpy().view(np.uint32)
    for a, b in ((0, chunk), (chunk, n)):
        own = ctx.classifier_forward(mesh, xp[a:b].contiguous()).cpu().numpy().view(np.uint32)
        assert np.array_equal(own, H[a:b])
    mesh.release()


@pytest.mark.parametrize("dim,B", [(2, 16), (2, 17), (2, 129), (2, 2000), (3, 17), (3, 130)])
def test_permuted_batch_gradient(ctx, dim, B):
    mesh = _mesh(ctx, dim)
    xp, lab, perm = _points(dim, B, B)
    g, loss = ctx.classifier_grad(mesh, xp, lab)
    gp, lp = ctx.classifier_grad(mesh, xp[perm].contiguous(), lab[perm].contiguous())
    assert bool(g.isfinite().all())
    assert abs(loss - lp) <= 1e-5 * loss
    assert float((g - gp).double().norm() / g.double().norm()) <= 2e-4
    again, _ = ctx.classifier_grad(mesh, xp, lab)
    assert np.array_equal(again.cpu().numpy().view(np.uint32), g.cpu().numpy().view(np.uint32))
    mesh.release()


@pytest.mark.parametrize("B", [152, 153, 305, 609])
def test_permuted_gradient_of_paired_windows(ctx, B):
    """The second layer's backward pass takes two windows a tile once every SM has
    one (152 SMs): one tile more, an odd window left over, a second tile per CTA.
    The bound is the permuted batch's above."""
    test_permuted_batch_gradient(ctx, 2, B)
