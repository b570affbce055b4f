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


def test_a_refused_predictor_grid_or_table(cs):
    """Each allocation of a coarser predictor grid, and of the table its grid
    velocity is interpolated with, refused in turn: the mesh keeps a grid it can
    use, and the call goes through once there is room. (Both had left a pointer
    behind that the next call would have used: one to freed memory, one null.)"""
    c = make_case("tg2d", n_side=41)
    roomy = cs.Context(0)
    mesh = roomy.upload_mesh(c.xyz, c.conn)
    base = roomy.memory_usage()[0]
    mesh.set_predictor_grid(3)
    want = roomy.grid_velocity(mesh, _dev(c.u), out=_dev(np.zeros((np.prod(mesh.info()["pred_grid"]), 2),
                                                                  np.float32))).cpu().numpy()
    asg = int(np.prod(mesh.info()["asg_grid"]))
    cells = int(np.prod(mesh.info()["pred_grid"]))
    mesh.set_predictor_grid(1)
    want1 = roomy.grid_velocity(mesh, _dev(c.u), out=_dev(np.zeros((asg, 2), np.float32))).cpu().numpy()
    roomy.close()
    table = 3 * 4 * cells            # node or weights
    for room in (0, 4 * cells, 4 * cells + table):
        ctx = cs.Context(0, hbm_budget=base + room)
        mesh = ctx.upload_mesh(c.xyz, c.conn)
        if room == 0:
            for _ in range(2):
                with pytest.raises(cs.CsError) as e:
                    mesh.set_predictor_grid(3)
                assert e.value.code == -2
                assert mesh.info()["pred_stride"] == 1
                assert list(mesh.info()["pred_grid"]) == list(mesh.info()["asg_grid"])
        else:
            mesh.set_predictor_grid(3)
        n = asg if room == 0 else cells
        out = _dev(np.zeros((n, 2), np.float32))
        for _ in range(2):
            with pytest.raises(cs.CsError) as e:
                ctx.grid_velocity(mesh, _dev(c.u), out=out)
            assert e.value.code == -2
        ctx.close()
    ctx = cs.Context(0, hbm_budget=base + 4 * cells + 2 * table)
    mesh = ctx.upload_mesh(c.xyz, c.conn)
    mesh.set_predictor_grid(3)
    out = ctx.grid_velocity(mesh, _dev(c.u), out=_dev(np.zeros((cells, 2), np.float32)))
    assert np.array_equal(out.cpu().numpy().view(np.uint32), want.view(np.uint32))
    ctx.close()
    # refused for the coarse grid's sake, then used with a released mesh's room
    ctx = cs.Context(0, hbm_budget=2 * base)
    other, mesh = ctx.upload_mesh(c.xyz, c.conn), ctx.upload_mesh(c.xyz, c.conn)
    with pytest.raises(cs.CsError):
        mesh.set_predictor_grid(3)
    other.release()
    out = ctx.grid_velocity(mesh, _dev(c.u), out=_dev(np.zeros((asg, 2), np.float32)))
    assert np.array_equal(out.cpu().numpy().view(np.uint32), want1.view(np.uint32))
    ctx.close()


def test_a_refused_grid_velocity_is_none(cs):
    """The grid velocity's buffer fits, the table it is computed with does not:
    the mesh has no grid velocity, and what reads it says so."""
    c = make_case("tg2d", n_side=41)
    probe = cs.Context(0)
    mesh = probe.upload_mesh(c.xyz, c.conn)
    base, asg = probe.memory_usage()[0], int(np.prod(mesh.info()["asg_grid"]))
    probe.close()
    ctx = cs.Context(0, hbm_budget=base + 2 * 8 * asg)       # velocity and prediction
    mesh = ctx.upload_mesh(c.xyz, c.conn)
    with pytest.raises(cs.CsError) as e:
        ctx.grid_velocity(mesh, _dev(c.u))
    assert e.value.code == -2
    with pytest.raises(cs.CsError) as e:
        ctx.windows(mesh, c.dt, B=4)
    assert e.value.code == -1 and "no grid velocity" in str(e.value)
    ctx.close()
