"""The workspaces of training and inference under an HBM budget.

The predictors have a layer-by-layer path (FP32 operands, and fewer than 16
rows) and fused ones, each with buffers that stay from call to call. A budget
that holds what the layer-by-layer path takes for a call has to hold the
fused path's call too, whatever calls of either kind came before: what a call
does not need is given back when memory runs out. Bar: no CS_ENOMEM, and the
bits of the same calls without a budget."""

import numpy as np
import pytest

from oracle import cnn
from workloads import make_case
from workloads.weights import init_classifier, init_weights

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cs():
    import paper_2412_18379_gb300 as cs
    from paper_2412_18379_gb300 import build
    build.build()
    return cs


class _Caller:
    """One context with a predictor or a classifier, and its gradient call."""

    def __init__(self, cs, kind, dim, budget=0):
        self.ctx, self.kind, self.dim = cs.Context(0, hbm_budget=budget), kind, dim
        if kind == "predictor":
            self.ctx.load_predictor(dim, init_weights(dim, 1))
        else:
            c = make_case("tg2d", n_side=41) if dim == 2 else make_case("abc3d", n_side=9)
            self.ctx.load_classifier(dim, init_classifier(dim, 1))
            self.mesh = self.ctx.upload_mesh(c.xyz, c.conn)

    def inputs(self, B):
        import torch
        gen = torch.Generator(device="cuda").manual_seed(B)
        if self.kind == "predictor":
            S = cnn.patch_size(self.dim)
            return (torch.randn((B, self.dim) + (S,) * self.dim, generator=gen, device="cuda"),
                    torch.randn((B, self.dim), generator=gen, device="cuda"))
        return (torch.rand((B, self.dim), dtype=torch.float64, generator=gen, device="cuda"),
                torch.randint(0, 81, (B,), dtype=torch.int32, generator=gen, device="cuda"))

    def grad(self, B, bf16=True):
        a, b = self.inputs(B)
        self.ctx.predictor_precision(bf16)
        try:
            g, _ = (self.ctx.predictor_grad(self.dim, a, b) if self.kind == "predictor"
                    else self.ctx.classifier_grad(self.mesh, a, b))
        finally:
            self.ctx.predictor_precision(True)
        return g.cpu().numpy().view(np.uint32)

    def forward(self, B):
        a, _ = self.inputs(B)
        out = (self.ctx.predictor_forward(self.dim, a) if self.kind == "predictor"
               else self.ctx.classifier_forward(self.mesh, a))
        return out.cpu().numpy().view(np.uint32)

    def used(self):
        return self.ctx.memory_usage()[0]


@pytest.mark.parametrize("kind", ["predictor", "classifier"])
@pytest.mark.parametrize("dim,B", [(2, 16), (2, 300), (3, 16), (3, 129), (3, 300)])
def test_the_fused_paths_fit_the_layers_budget(cs, kind, dim, B):
    roomy = _Caller(cs, kind, dim)
    want = {bf16: roomy.grad(B, bf16) for bf16 in (False, True)}
    want[15] = roomy.grad(15)
    want["forward"] = roomy.forward(B)
    roomy.ctx.close()
    probe = _Caller(cs, kind, dim)
    probe.grad(B, bf16=False)
    budget = probe.used()
    probe.ctx.close()
    tight = _Caller(cs, kind, dim, budget)
    for _ in range(2):      # the fused path, the layers' path on what it left, and back
        assert np.array_equal(tight.grad(B), want[True])
        assert np.array_equal(tight.grad(15), want[15])
        assert np.array_equal(tight.grad(B), want[True])
        assert np.array_equal(tight.grad(B, bf16=False), want[False])
        assert np.array_equal(tight.forward(B), want["forward"])
    assert tight.used() <= budget
    tight.ctx.close()


def test_other_allocations_take_idle_workspaces(cs):
    """A mesh that fits beside the weights, not beside the workspaces of a call
    before: they are given back for it, and the next call makes them again."""
    one = _Caller(cs, "predictor", 2)
    weights = one.used()
    want = one.grad(4096)
    work = one.used() - weights
    c = make_case("tg2d", n_side=101)
    mesh = one.ctx.upload_mesh(c.xyz, c.conn).info()["device_bytes"]
    one.ctx.close()
    tight = _Caller(cs, "predictor", 2, weights + max(mesh, work) + 1024)
    assert np.array_equal(tight.grad(4096), want)
    m = tight.ctx.upload_mesh(c.xyz, c.conn)
    assert tight.used() == weights + mesh
    m.release()
    assert np.array_equal(tight.grad(4096), want)
    # what a call needs is never given back: too large a batch is refused
    with pytest.raises(cs.CsError) as e:
        tight.grad(40960)
    assert e.value.code == -2
    assert np.array_equal(tight.grad(4096), want)
    tight.ctx.close()


def test_a_layers_call_leaves_the_serving_tiles(cs):
    """With the CUDA-core engine, serving predicts in 3-D into a workspace that a
    layer-by-layer call (fewer than 16 rows) had freed as it grew its own."""
    import torch
    c = make_case("abc3d", n_side=13)
    ctx = cs.Context(0)
    ctx.load_predictor(3, init_weights(3, 1))
    ctx.predictor_engine("tiles")
    mesh = ctx.upload_mesh(c.xyz, c.conn)
    field = ctx.upload_field(mesh, c.u)
    x, u = (torch.from_numpy(np.ascontiguousarray(a)).pin_memory() for a in (c.x, c.u))
    start = torch.from_numpy(mesh.node_start_elements()).pin_memory()
    win = torch.randn((8, 3, 7, 7, 7), device="cuda")
    tgt = torch.randn((8, 3), device="cuda")
    torch.cuda.synchronize()
    ctx.serve_start(slots=2, arena_bytes=64 << 20)
    try:
        results = []
        for _ in range(2):
            ticket, out = ctx.submit(mesh, x, u, c.dt, start=start, mode="cnn", field=field)
            assert ctx.wait(ticket) == 1              # started by the predictor
            results.append({k: v.clone() for k, v in out.items()})
            ctx.predictor_grad(3, win, tgt)
        for k in results[0]:
            assert torch.equal(results[0][k], results[1][k]), k
    finally:
        ctx.serve_stop()
    ctx.close()
