"""The fused training kernels at the edges of their tiles.

A batch is cut into tiles of whole windows (5 per tile in the 2-D network's
second layer, one per CTA and SM in its last); the batch sizes leave one row
over, fill a tile exactly, or limit the windows of a tile by shared memory
(8200 in 3-D). Each window's output depends on that window alone, so permuting
the batch permutes the outputs bit for bit. The gradients are sums over the
batch: a permutation moves rows between tiles and CTAs and changes only the
order of FP32 sums. A sum of N terms of random sign errs by about sqrt(N)
2^-24 of its terms' size, and the sum itself may be as small as the terms'
root sum of squares: for N <= 8200 * 125 positions 1e3 * 6e-8 = 6e-5, allowed
2e-4 in norm, while a lost or doubled row would show at 1 / B >= 1.2e-4 of
the coherent part per row and at its full size in batches of 16 and 17.
"""

import numpy as np
import pytest

from oracle import cnn
from workloads.weights import init_weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2412_18379_gb300 as cs
    from paper_2412_18379_gb300 import build
    build.build()
    c = cs.Context(0)
    yield c
    c.close()


def _pairs(dim, B, seed):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    S = cnn.patch_size(dim)
    win = torch.randn((B, dim) + (S,) * dim, generator=gen, device="cuda")
    tgt = torch.randn((B, dim), generator=gen, device="cuda")
    return win, tgt, torch.randperm(B, generator=gen, device="cuda")


@pytest.mark.parametrize("dim,B", [(2, 16), (2, 17), (2, 761), (2, 4096), (2, 9729),
                                   (3, 16), (3, 17), (3, 609), (3, 8200)])
def test_a_permuted_batch(ctx, dim, B):
    ctx.load_predictor(dim, init_weights(dim, 23))
    win, tgt, perm = _pairs(dim, B, 100 * dim + B)
    out = ctx.predictor_forward(dim, win)
    # chunks of 8192: within one chunk the outputs are the same bits
    n = min(B, 8192)
    head = win[:n][perm[perm < n]].contiguous()
    if n == B:
        assert np.array_equal(ctx.predictor_forward(dim, head).cpu().numpy().view(np.uint32),
                              out[perm].cpu().numpy().view(np.uint32))
    g, loss = ctx.predictor_grad(dim, win, tgt)
    gp, lp = ctx.predictor_grad(dim, win[perm].contiguous(), tgt[perm].contiguous())
    ctx.device_status()
    assert abs(loss - lp) <= 1e-5 * loss
    assert float((g - gp).double().norm() / g.double().norm()) <= 2e-4
    # the same call again gives the same bits
    again, _ = ctx.predictor_grad(dim, win, tgt)
    assert np.array_equal(again.cpu().numpy().view(np.uint32), g.cpu().numpy().view(np.uint32))


@pytest.mark.parametrize("dim,B", [(2, 17), (2, 153), (3, 17)])
def test_a_repeated_batch(ctx, dim, B):
    """The mean over a batch is the mean over eight copies of it. The loss
    gradient's factor 1 / B changes by 8, a power of two, so every BF16 value of
    the backward pass is scaled exactly and only the order of FP32 sums
    differs (sizes at which a 3-D convolution's K is split alike in both
    batches): sqrt(8 * 153 * 49) 2^-24 = 1.5e-5 of the terms, allowed 2e-4 in
    norm as above."""
    ctx.load_predictor(dim, init_weights(dim, 7))
    win, tgt, _ = _pairs(dim, B, B)
    rep = (8,) + (1,) * (win.dim() - 1)
    g, loss = ctx.predictor_grad(dim, win, tgt)
    g8, loss8 = ctx.predictor_grad(dim, win.repeat(rep).contiguous(), tgt.repeat(8, 1).contiguous())
    ctx.device_status()
    assert abs(loss - loss8) <= 1e-5 * loss
    assert float((g - g8).double().norm() / g.double().norm()) <= 2e-4
