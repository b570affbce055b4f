"""The device memory a mesh takes, and walks that end at a node within it.

A budget that held a mesh and what is uploaded after it has to go on holding
them: an upload takes the arrays below and nothing for speed's sake beside
them, whatever room there is. Bar: their bytes, and the oracle's hosts, path
lengths and statuses bit for bit under a budget without a byte to spare."""

import numpy as np
import pytest

import oracle
from workloads import make_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cs():
    import paper_2412_18379_gb300 as cs
    from paper_2412_18379_gb300 import build
    build.build()
    return cs


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _mesh_bytes(info):
    d, n_v, n_e = info["dim"], info["n_vertices"], info["n_elements"]
    asg = int(np.prod(info["asg_grid"][:d]))
    buckets = int(np.prod(info["bucket_grid"][:d]))
    records = n_e * ((48 + 48) if d == 2 else (80 + 96))     # walk, exact
    per_element = n_e * (4 + 4 * (d + 1) + 8 * d)            # iperm, conn, centroid
    per_vertex = n_v * (4 + 8 * d)                           # plain start, xyz
    index = 4 * (buckets + 1) + 4 * info["bucket_items"]
    grid = asg * (4 + 8 * d + 8 * d)                         # seed, pool, pool as floats
    return records + per_element + per_vertex + index + grid


@pytest.mark.parametrize("name,n_side,drop", [("tg2d", 21, 0), ("tg2d", 21, 1), ("abc3d", 9, 0),
                                              ("abc3d", 9, 1)])
def test_mesh_bytes(cs, name, n_side, drop):
    """drop: an odd number of elements (one left out, its neighbours' faces then
    on the boundary)."""
    c = make_case(name, n_side=n_side)
    conn = c.conn[:len(c.conn) - drop]
    assert len(conn) % 2 == drop
    ctx = cs.Context(0)
    info = ctx.upload_mesh(c.xyz, conn).info()
    assert info["device_bytes"] == _mesh_bytes(info)
    assert ctx.memory_usage()[0] == info["device_bytes"]
    ctx.close()


def test_an_exact_budget(cs):
    """A mesh, its field and a prediction in the bytes they take, then walks of
    nodes at rest and around them."""
    import torch
    from workloads.weights import init_weights
    c = make_case("sphere3d", n_side=13)
    probe = cs.Context(0)
    mesh = probe.upload_mesh(c.xyz, c.conn)
    mesh_bytes = _mesh_bytes(mesh.info())
    probe.load_predictor(3, init_weights(3, 1))
    field = probe.upload_field(mesh, c.u)
    probe.track(mesh, _dev(c.x), _dev(c.u), c.dt, mode="cnn", field=field)
    torch.cuda.synchronize()
    rest = probe.memory_usage()[0] - mesh.info()["device_bytes"]
    probe.close()

    ctx = cs.Context(0, hbm_budget=mesh_bytes + rest)
    mesh = ctx.upload_mesh(c.xyz, c.conn)
    assert not ctx.lib.cs_last_error(ctx.h)
    ctx.load_predictor(3, init_weights(3, 1))
    field = ctx.upload_field(mesh, c.u)
    om = oracle.Mesh(c.xyz, c.conn, grid=mesh.info()["asg_grid"])
    rng = np.random.default_rng(3)
    for delta in (0.0, 1e-16, 1e-15, 1e-12):
        u = rng.standard_normal(c.x.shape)
        u *= delta / np.linalg.norm(u, axis=1, keepdims=True)
        want = om.track(c.x, u, 1.0)
        out = ctx.track(mesh, _dev(c.x), _dev(u), 1.0)
        for k in ("host", "path_len", "status"):
            assert np.array_equal(out[k].cpu().numpy(), want[k]), (delta, k)
        out = ctx.track(mesh, _dev(c.x), _dev(u), 1.0, mode="cnn", field=field)
        assert np.array_equal(out["host"].cpu().numpy(), want["host"]), delta
    assert ctx.memory_usage()[0] <= mesh_bytes + rest
    ctx.close()
