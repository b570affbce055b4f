"""Particles at rest, or almost, at a node: their host comes from the mesh's
table of the points around each vertex (search.cu) instead of the exact
search. Bar: the oracle's hosts, path lengths and statuses bit for bit, at the
vertex itself and at distances from it below, around and beyond the radius
within which the table answers (about 1e-16 to 1e-15 here; the tolerance of
containment is 1e-12)."""

import numpy as np
import pytest

import oracle
from workloads import element_node_particles, make_case

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    import paper_2412_18379_gb300 as cs
    from paper_2412_18379_gb300 import build
    build.build()
    c = cs.Context(0)
    yield c
    c.close()


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("name,n_side", [("tg2d", 41), ("hole2d", 61), ("abc3d", 9),
                                         ("sphere3d", 25)])
def test_particles_at_rest_at_nodes(ctx, name, n_side):
    c = make_case(name, n_side=n_side)
    mesh = ctx.upload_mesh(c.xyz, c.conn)
    om = oracle.Mesh(c.xyz, c.conn, grid=mesh.info()["asg_grid"])
    rng = np.random.default_rng(n_side)
    pairs = element_node_particles(c)
    for delta in (0.0, 1e-18, 1e-16, 3e-16, 1e-15, 1e-14, 1e-13, 1e-12, 1e-11, 1e-9):
        for x, start in ((c.x, None), (pairs[0], pairs[2])):
            u = rng.standard_normal(x.shape)
            u *= delta / np.linalg.norm(u, axis=1, keepdims=True)
            out = ctx.track(mesh, _dev(x), _dev(u), 1.0,
                            start=None if start is None else _dev(start))
            want = om.track(x, u, 1.0, start=start)
            for k in ("host", "path_len", "status"):
                assert np.array_equal(out[k].cpu().numpy(), want[k]), (delta, k)
    mesh.release()
