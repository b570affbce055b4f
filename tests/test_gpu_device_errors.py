"""The device error flag at the end of the predictor's synchronous calls.

A kernel whose bounded wait gives up writes no results; the sums and copies
behind it would take what an earlier call left in their place. The flag is
raised here as the library's own test hook does it: a grid prediction, which
does not synchronise, waits for a device flag that nothing sets and gives up.
The next synchronous call has to report it, and the one after that gives the
bits it gave before."""

import numpy as np
import pytest

from oracle import cnn
from workloads import make_case
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


def _give_up(ctx, mesh, dt):
    """A grid prediction whose wait has run out, the device idle again."""
    import torch
    out = torch.empty((int(np.prod(mesh.info()["pred_grid"])), mesh.dim), device="cuda")
    ctx.debug_hold_predictor(True)
    try:
        ctx.predict(mesh, dt, out=out)
        torch.cuda.synchronize()
    finally:
        ctx.debug_hold_predictor(False)


@pytest.mark.parametrize("dim,B", [(2, 7), (2, 40), (3, 7), (3, 40)])
def test_a_given_up_wait_is_reported(ctx, dim, B):
    """7 rows take the layer-by-layer path, 40 the fused one."""
    import torch
    import paper_2412_18379_gb300 as cs
    c = make_case("tg2d", n_side=41) if dim == 2 else make_case("abc3d", n_side=9)
    ctx.load_predictor(dim, init_weights(dim, 3))
    mesh = ctx.upload_mesh(c.xyz, c.conn)
    ctx.grid_velocity(mesh, torch.from_numpy(np.ascontiguousarray(c.u)).cuda())
    gen = torch.Generator(device="cuda").manual_seed(B)
    win = torch.randn((B, dim) + (cnn.patch_size(dim),) * dim, generator=gen, device="cuda")
    tgt = torch.randn((B, dim), generator=gen, device="cuda")
    calls = {"forward": lambda: ctx.predictor_forward(dim, win).cpu().numpy(),
             "grad": lambda: ctx.predictor_grad(dim, win, tgt)[0].cpu().numpy()}
    for name, call in calls.items():
        want = call()
        _give_up(ctx, mesh, c.dt)
        with pytest.raises(cs.CsError) as e:
            call()
        assert e.value.code == -8 and "gave up" in str(e.value), name
        assert np.array_equal(call().view(np.uint32), want.view(np.uint32)), name
    weights = ctx.save_predictor(dim)
    _give_up(ctx, mesh, c.dt)
    with pytest.raises(cs.CsError) as e:
        ctx.train(dim, win, tgt, batch=B, steps=2)
    assert e.value.code == -8
    assert np.array_equal(ctx.save_predictor(dim), weights)
    ctx.train(dim, win, tgt, batch=B, steps=2)
    assert not np.array_equal(ctx.save_predictor(dim), weights)
    mesh.release()
