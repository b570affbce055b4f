"""The calls that a user of the library makes, as measurable cases.

A solver keeps one context and a resident mesh and calls the library every
time step with a new velocity; a training program calls the gradients of one
batch after another; the classifier evaluates every departure point. Each case
is one such call through the public binding, at sizes of the meshes that the
repository's benchmark, serving workload and tests use: 2.6 thousand to a
million nodes in 2-D, a few thousand to half a million in 3-D, batches of a few
hundred to 8192 training pairs.

What a program keeps between calls (the context, the mesh on the device, the
loaded networks) is made once per process and shared; what changes from step
to step (the velocity field, the time step, the batch) is made by prepare()
from the seed.
"""

import functools
import math
import weakref

import numpy as np
import torch

import paper_2412_18379_gb300 as cs

DEV = "cuda:0"


# --------------------------------------------------------------------------
# the cases
# --------------------------------------------------------------------------

def listed():
    return [
        # a time step of a small solver: one call's latency
        {"name": "nodes-sns-2d-small", "kind": "nodes", "dim": 2, "n_side": 51, "mode": "sns",
         "cfl": 2.0},
        # a time step of the two-million-triangle mesh, plain SNS and CNN-SNS
        {"name": "nodes-sns-2d", "kind": "nodes", "dim": 2, "n_side": 1001, "mode": "sns",
         "cfl": 8.0},
        {"name": "nodes-cnn-2d", "kind": "nodes", "dim": 2, "n_side": 1001, "mode": "cnn",
         "cfl": 8.0},
        # the same through host memory, copies included, on a middle mesh of odd size
        {"name": "host-cnn-2d", "kind": "host", "dim": 2, "n_side": 487, "mode": "cnn",
         "cfl": 8.0},
        # characteristic tracing of a finite element step: a particle per
        # (element, node) pair, each starting from its element
        {"name": "pairs-sns-3d", "kind": "pairs", "dim": 3, "n_side": 41, "mode": "sns",
         "cfl": 4.0},
        # a time step in 3-D with the velocity resident as a field
        {"name": "field-cnn-3d", "kind": "field", "dim": 3, "n_side": 75, "mode": "cnn",
         "cfl": 8.0},
        # the start predictor over a fine grid: resample, then the network on every cell
        {"name": "predict-2d", "kind": "predict", "dim": 2, "n_side": 701, "stride": 1},
        # the gradients of one training batch of the start predictor
        {"name": "grad-2d", "kind": "grad", "dim": 2, "batch": 4096},
        {"name": "grad-3d", "kind": "grad", "dim": 3, "batch": 2048},
        # the paper's classifier on every departure point of a step, and its training
        {"name": "classify-2d", "kind": "classify", "dim": 2, "n_side": 401, "n": 160801},
        {"name": "classify-3d", "kind": "classify", "dim": 3, "n_side": 27, "n": 19683},
        {"name": "classify-grad-2d", "kind": "classify-grad", "dim": 2, "n_side": 201,
         "batch": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["nodes", "nodes", "host", "pairs", "field", "predict", "grad", "grad",
                       "classify", "classify", "classify-grad"])
    dim = rng.choice([2, 3])
    if kind in ("nodes", "host", "field"):
        side = _log_int(rng, 33, 1001) if dim == 2 else _log_int(rng, 15, 75)
        modes = ["cnn"] if kind == "field" else ["sns", "cnn", "asg"]
        return {"kind": kind, "dim": dim, "n_side": side, "mode": rng.choice(modes),
                "cfl": round(rng.uniform(1.0, 12.0), 2)}
    if kind == "pairs":
        side = _log_int(rng, 21, 420) if dim == 2 else _log_int(rng, 9, 41)
        return {"kind": kind, "dim": dim, "n_side": side, "mode": rng.choice(["sns", "asg"]),
                "cfl": round(rng.uniform(1.0, 6.0), 2)}
    if kind == "predict":
        side = _log_int(rng, 60, 701) if dim == 2 else _log_int(rng, 17, 60)
        return {"kind": kind, "dim": dim, "n_side": side, "stride": rng.choice([1, 3, 5])}
    if kind == "grad":
        return {"kind": kind, "dim": dim,
                "batch": _log_int(rng, 256, 8192 if dim == 2 else 4096)}
    if kind == "classify":
        side = _log_int(rng, 33, 401) if dim == 2 else _log_int(rng, 11, 41)
        return {"kind": kind, "dim": dim, "n_side": side,
                "n": _log_int(rng, 500, 160000 if dim == 2 else 19000)}
    side = _log_int(rng, 33, 201) if dim == 2 else _log_int(rng, 11, 27)
    return {"kind": kind, "dim": dim, "n_side": side,
            "batch": _log_int(rng, 256, 4096 if dim == 2 else 512)}


# --------------------------------------------------------------------------
# meshes: jittered lattices of the unit square or cube, two triangles per
# square, six Kuhn tetrahedra per cube (the jitter is small enough that no
# element can turn over)
# --------------------------------------------------------------------------

@functools.lru_cache(maxsize=2)
def _lattice(dim, n):
    """(xyz [n_v, dim], conn [n_e, dim + 1]) with node id (iz n + iy) n + ix."""
    h = 1.0 / (n - 1)
    g = np.linspace(0.0, 1.0, n)
    rng = np.random.default_rng(40 + dim)
    if dim == 2:
        Y, X = np.meshgrid(g, g, indexing="ij")
        xyz = np.stack([X.ravel(), Y.ravel()], axis=1)
        jitter = 0.15
        ix, iy = np.tile(np.arange(n - 1), n - 1), np.repeat(np.arange(n - 1), n - 1)
        v = iy * n + ix
        conn = np.stack([np.stack([v, v + 1, v + n + 1], axis=1),
                         np.stack([v, v + n + 1, v + n], axis=1)], axis=1)
    else:
        Z, Y, X = np.meshgrid(g, g, g, indexing="ij")
        xyz = np.stack([X.ravel(), Y.ravel(), Z.ravel()], axis=1)
        jitter = 0.05
        i = np.arange(n - 1)
        v = ((i[:, None, None] * n + i[None, :, None]) * n + i[None, None, :]).ravel()
        step = (1, n, n * n)
        tets = []
        for a, b in ((0, 1), (0, 2), (1, 0), (1, 2), (2, 0), (2, 1)):
            e1 = v + step[a]
            tets.append(np.stack([v, e1, e1 + step[b], v + sum(step)], axis=1))
        conn = np.stack(tets, axis=1)
    inner = ((xyz > 0.5 * h) & (xyz < 1.0 - 0.5 * h)).all(axis=1)
    xyz = xyz + np.where(inner[:, None], rng.uniform(-jitter * h, jitter * h, xyz.shape), 0.0)
    return np.ascontiguousarray(xyz), np.ascontiguousarray(
        conn.reshape(-1, dim + 1).astype(np.int32))


class _Program:
    """A context with its networks loaded, and its resident meshes."""

    def __init__(self, role):
        self.ctx = cs.Context(0)
        self.meshes = {}
        for dim in (2, 3):
            if role == "track":
                self.ctx.load_predictor(dim, _displacement_weights(dim))
            elif role == "train":
                self.ctx.load_predictor(dim, _initial(_predictor_layers(dim), 10 + dim))
            else:
                self.ctx.load_classifier(dim, _initial(_classifier_layers(dim), 20 + dim))

    def mesh(self, dim, n, stride=1):
        """The resident mesh and its vertices on the device."""
        key = (dim, n, stride)
        if key not in self.meshes:
            while len(self.meshes) >= 2:
                self.meshes.pop(next(iter(self.meshes)))[0].release()
            xyz, conn = _lattice(dim, n)
            m = self.ctx.upload_mesh(xyz, conn)
            if stride != 1:
                m.set_predictor_grid(stride)
            self.meshes[key] = (m, torch.from_numpy(xyz).to(DEV))
        return self.meshes[key]


@functools.lru_cache(maxsize=None)
def _program(role):
    return _Program(role)


# --------------------------------------------------------------------------
# networks (flat float32 parameters; W then b of each layer)
# --------------------------------------------------------------------------

def _predictor_layers(dim):
    taps, n_conv = (9, 4) if dim == 2 else (27, 3)
    shapes = [(32, dim if l == 0 else 32, taps) for l in range(n_conv)]
    return shapes + [(256, 32), (dim, 256)]


def _classifier_layers(dim):
    W, taps = (9, 9) if dim == 2 else (7, 27)
    return [(32, dim, taps), (32, 32, taps), (256, dim), (256, 256),
            (512, 32 * (W // 2) ** dim + 256), (W ** dim, 512)]


def _initial(shapes, seed):
    """He-normal weights and zero biases: a network as its training begins."""
    rng = np.random.default_rng(seed)
    parts = []
    for s in shapes:
        parts += [rng.standard_normal(s).ravel() * math.sqrt(2.0 / np.prod(s[1:])),
                  np.zeros(s[0])]
    return np.concatenate(parts).astype(np.float32)


def _displacement_weights(dim):
    """A predictor that knows its task: 2 dim channels carry +-u of the centre
    cell to the output -u (the first-order displacement); the others hold a
    small random network, whose share of the output is about a hundredth."""
    rng = np.random.default_rng(30 + dim)
    shapes = _predictor_layers(dim)
    centre, c = (4 if dim == 2 else 13), 2 * dim
    parts = []
    for l, s in enumerate(shapes):
        W = rng.standard_normal(s) * math.sqrt(2.0 / np.prod(s[1:]))
        if l < len(shapes) - 1:
            W[:c] = 0.0
        if l == 0:
            for k in range(dim):
                W[2 * k, k, centre], W[2 * k + 1, k, centre] = 1.0, -1.0
        elif l < len(shapes) - 2:
            W[np.arange(c), np.arange(c), centre] = 1.0
        elif l == len(shapes) - 2:
            W[np.arange(c), np.arange(c)] = 1.0
        else:
            W *= 0.01
            W[:, :c] = 0.0
            for k in range(dim):
                W[k, 2 * k], W[k, 2 * k + 1] = -1.0, 1.0
        parts += [W.ravel(), np.zeros(s[0])]
    return np.concatenate(parts).astype(np.float32)


def _layers(flat, shapes):
    """[(W, b)] in 64 bits on the device from the flat parameters."""
    out, o = [], 0
    flat = torch.from_numpy(flat.astype(np.float64)).to(DEV)
    for s in shapes:
        n = int(np.prod(s))
        W = flat[o:o + n].reshape(s)
        if len(s) == 3:
            W = W.reshape(s[0], s[1], *((3,) * (2 if s[2] == 9 else 3)))
        out.append((W, flat[o + n:o + n + s[0]]))
        o += n + s[0]
    return out


# --------------------------------------------------------------------------
# velocity fields
# --------------------------------------------------------------------------

def _modes(p, seed):
    """A random flow at points p [..., dim] (64 bits): eight Fourier modes of a
    stream function (2-D) or vector potential (3-D), zero flow through the
    walls of the unit box."""
    dim = p.shape[-1]
    rng = np.random.default_rng(seed)
    a = rng.standard_normal((8, 1 if dim == 2 else 3))
    m = rng.integers(1, 5, (8, dim))
    u = [torch.zeros_like(p[..., 0]) for _ in range(dim)]
    for j in range(8):
        t = [math.pi * float(m[j, k]) * p[..., k] for k in range(dim)]
        s, c = [torch.sin(v) for v in t], [torch.cos(v) for v in t]
        if dim == 2:
            u[0] = u[0] + float(a[j, 0] * m[j, 1]) * s[0] * c[1]
            u[1] = u[1] - float(a[j, 0] * m[j, 0]) * c[0] * s[1]
        else:
            dx = float(m[j, 0]) * c[0] * s[1] * s[2]
            dy = float(m[j, 1]) * s[0] * c[1] * s[2]
            dz = float(m[j, 2]) * s[0] * s[1] * c[2]
            a0, a1, a2 = (float(v) for v in a[j])
            u[0] = u[0] + a2 * dy - a1 * dz
            u[1] = u[1] + a0 * dz - a2 * dx
            u[2] = u[2] + a1 * dx - a0 * dy
    return torch.stack(u, dim=-1).contiguous()


def _dt(u, n_side, cfl):
    return cfl / (n_side - 1) / float(u.square().sum(-1).max().sqrt())


def _linear_flow(dim, seed):
    """(A, b) of a flow u = A x + b: a rotation, a strain and a drift."""
    rng = np.random.default_rng(seed)
    return rng.standard_normal((dim, dim)), 0.3 * rng.standard_normal(dim)


def _windows(dim, batch, seed):
    """Training pairs: windows of u dt / s around random cells of a grid of
    200^2 or 20^3 predictor cells (zero outside it), four flows at CFL 2 to
    16, and the displacement -u dt / s of a particle in the cell."""
    rng = np.random.default_rng(seed)
    S, g = (9, 200) if dim == 2 else (7, 20)
    s = 1.0 / g
    cell = rng.integers(0, g, (batch, dim))
    off = np.stack(np.meshgrid(*([np.arange(S) - S // 2] * dim), indexing="ij")[::-1], axis=-1)
    cc = torch.from_numpy(cell.reshape((batch,) + (1,) * dim + (dim,)) + off).to(DEV)
    inside = ((cc >= 0) & (cc < g)).all(-1)
    at = torch.from_numpy((cell + rng.random((batch, dim))) * s).to(DEV)
    win = torch.empty((batch, dim) + (S,) * dim, dtype=torch.float32, device=DEV)
    tgt = torch.empty((batch, dim), dtype=torch.float32, device=DEV)
    for f in range(4):
        part = slice(f * batch // 4, (f + 1) * batch // 4)
        field = 4 * seed + f
        scale = float(rng.uniform(2.0, 16.0)) / 5.0 / 8.0     # dt / s: CFL in fifths of a cell
        u = _modes((cc[part].double() + 0.5) * s, field) * scale
        u = torch.where(inside[part][..., None], u, torch.zeros_like(u))
        win[part] = u.movedim(-1, 1).float()
        tgt[part] = (-scale * _modes(at[part], field)).float()
    return win, tgt


def _departures(dim, n_side, n, seed):
    """n departure points x - u dt of random particles at CFL 8."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    x = torch.rand((n, dim), dtype=torch.float64, device=DEV, generator=gen)
    u = _modes(x, seed)
    return (x - u * _dt(u, n_side, 8.0)).contiguous(), gen


def _labels(dim, n_side, xp, gen):
    """Window cells (x fastest) of points up to half a cell from x_p, as the
    centroid of x_p's host lies."""
    g, W = n_side - 1, 9 if dim == 2 else 7
    near = xp * g + torch.rand(xp.shape, dtype=torch.float64, device=DEV, generator=gen) - 0.5
    c0 = torch.floor(xp * g).clamp(0, g - 1)
    rel = (torch.floor(near).clamp(0, g - 1) - c0 + W // 2).clamp(0, W - 1).long()
    cls = rel[:, dim - 1]
    for k in range(dim - 2, -1, -1):
        cls = cls * W + rel[:, k]
    return cls.to(torch.int32).contiguous()


# --------------------------------------------------------------------------
# prepare and run
# --------------------------------------------------------------------------

def _outputs(n, **kw):
    return {"host": torch.empty(n, dtype=torch.int32, **kw),
            "path_len": torch.empty(n, dtype=torch.int32, **kw),
            "status": torch.empty(n, dtype=torch.uint8, **kw)}


def prepare(case, seed):
    kind, dim = case["kind"], case["dim"]
    s = {"kind": kind, "dim": dim, "mode": case.get("mode")}
    if kind == "grad":
        s["ctx"] = _program("train").ctx
        s["windows"], s["targets"] = _windows(dim, case["batch"], seed)
        return s
    if kind in ("classify", "classify-grad"):
        prog = _program("classify")
        s["ctx"], s["mesh"] = prog.ctx, prog.mesh(dim, case["n_side"])[0]
        n = case["n"] if kind == "classify" else case["batch"]
        s["xp"], gen = _departures(dim, case["n_side"], n, seed)
        if kind == "classify-grad":
            s["labels"] = _labels(dim, case["n_side"], s["xp"], gen)
        return s
    prog = _program("track")
    # CNN-SNS runs its predictor on cells of 5 ASG cells per axis, the benchmark's grid
    stride = case.get("stride", 5)
    s["ctx"] = prog.ctx
    s["mesh"], x = prog.mesh(dim, case["n_side"], stride)
    if kind == "predict":
        A, b = _linear_flow(dim, seed)
        s["u"] = (x @ torch.from_numpy(A.T.copy()).to(DEV) + torch.from_numpy(b).to(DEV)).contiguous()
        s["dt"] = _dt(s["u"], case["n_side"], 8.0)
        cells = int(np.prod([(case["n_side"] - 1) // stride] * dim))
        s["out"] = torch.empty((cells, dim), dtype=torch.float32, device=DEV)
        return s
    u = _modes(x, seed)
    s["dt"] = _dt(u, case["n_side"], case["cfl"])
    if kind == "pairs":
        conn = torch.from_numpy(_lattice(dim, case["n_side"])[1]).to(DEV).long().reshape(-1)
        s["x"], s["u"] = x[conn].contiguous(), u[conn].contiguous()
        s["start"] = torch.arange(conn.numel() // (dim + 1), dtype=torch.int32,
                                  device=DEV).repeat_interleave(dim + 1)
    elif kind == "host":
        s["u"] = u.cpu().pin_memory()
        s["out"] = _outputs(x.shape[0], pin_memory=True)
        return s
    else:
        s["x"], s["u"] = x, u
        if kind == "field":
            s["field"] = s["ctx"].upload_field(s["mesh"], u)
            weakref.finalize(u, _release, s["field"]).atexit = False
    s["out"] = _outputs(s["x"].shape[0], device=DEV)
    return s


def _release(field):
    if field.mesh.id is not None:      # a released mesh has taken its fields along
        field.release()


def run(state):
    s = state
    ctx, kind = s["ctx"], s["kind"]
    if kind in ("nodes", "pairs", "field"):
        return ctx.track(s["mesh"], s["x"], s["u"], s["dt"], start=s.get("start"),
                         mode=s["mode"], out=s["out"], field=s.get("field"))
    if kind == "host":
        return ctx.track_nodes_host(s["mesh"], s["u"], s["dt"], mode=s["mode"], out=s["out"])
    if kind == "predict":
        ctx.grid_velocity(s["mesh"], s["u"])
        return ctx.predict(s["mesh"], s["dt"], out=s["out"])
    if kind == "grad":
        return ctx.predictor_grad(s["dim"], s["windows"], s["targets"])
    if kind == "classify":
        return ctx.classifier_forward(s["mesh"], s["xp"])
    return ctx.classifier_grad(s["mesh"], s["xp"], s["labels"])


# --------------------------------------------------------------------------
# what a pass cannot do without
# --------------------------------------------------------------------------

def _macs(shapes, positions):
    return sum(int(np.prod(s)) * p for s, p in zip(shapes, positions))


def work(case):
    kind, dim = case["kind"], case["dim"]
    if kind == "grad":
        S = 9 if dim == 2 else 7
        pos = [(S - 2 * l) ** dim for l in range(1, 5 if dim == 2 else 4)] + [1, 1]
        shapes = _predictor_layers(dim)
        params = sum(int(np.prod(t)) + t[0] for t in shapes)
        return {"flops": 6.0 * _macs(shapes, pos) * case["batch"],
                "bytes": 4.0 * case["batch"] * dim * (S ** dim + 1) + 8.0 * params}
    if kind in ("classify", "classify-grad"):
        W = 9 if dim == 2 else 7
        shapes = _classifier_layers(dim)
        macs = _macs(shapes, [W ** dim, W ** dim, 1, 1, 1, 1])
        params = sum(int(np.prod(t)) + t[0] for t in shapes)
        if kind == "classify":
            return {"flops": 2.0 * macs * case["n"],
                    "bytes": case["n"] * (8.0 * dim + 4.0 * W ** dim) + 4.0 * params}
        return {"flops": 6.0 * macs * case["batch"],
                "bytes": case["batch"] * (8.0 * dim + 4.0) + 8.0 * params}
    n_side = case["n_side"]
    nodes = n_side ** dim
    elements = (n_side - 1) ** dim * (2 if dim == 2 else 6)
    stride = case.get("stride", 5)
    cells = ((n_side - 1) // stride) ** dim
    net = 2.0 * _macs(_predictor_layers(dim), [1] * 6) * cells
    if kind == "predict":
        return {"flops": net, "bytes": 8.0 * dim * nodes + 4.0 * dim * cells}
    n = elements * (dim + 1) if kind == "pairs" else nodes
    record = 48.0 if dim == 2 else 80.0      # one element: vertex, matrix, neighbours
    # x, u, start and the three outputs of a particle, and its host element once
    return {"flops": net if case["mode"] == "cnn" else 0.0,
            "bytes": n * (16.0 * dim + 4.0 + 9.0) + min(n, elements) * record}


# --------------------------------------------------------------------------
# the networks in 64 bits
# --------------------------------------------------------------------------

def _conv(x, W, b, pad=0):
    f = torch.nn.functional.conv2d if W.dim() == 4 else torch.nn.functional.conv3d
    return f(x, W, b, padding=pad)


def _predictor(x, layers):
    """x [B, dim, ...] through valid convolutions; [B, 256-wide head] per position."""
    for W, b in layers[:-2]:
        x = _conv(x, W, b).relu()
    (W1, b1), (W2, b2) = layers[-2:]
    x = x.movedim(1, -1)
    return (x @ W1.T + b1).relu() @ W2.T + b2


def _classifier(win, off, layers):
    (W1, b1), (W2, b2), (X1, c1), (X2, c2), (F, f), (L, l) = layers
    dim = off.shape[1]
    pool = torch.nn.functional.avg_pool2d if dim == 2 else torch.nn.functional.avg_pool3d
    p = pool(_conv(_conv(win, W1, b1, 1).relu(), W2, b2, 1).relu(), 2)
    y = ((off @ X1.T + c1).relu() @ X2.T + c2).relu()
    return (torch.cat([p.flatten(1), y], dim=1) @ F.T + f).relu() @ L.T + l


def _pooled_centroids(dim, n_side):
    """Mean element centroid per grid cell, the cell's centre where it has none
    ([g^dim, dim], x fastest); the grid is the lattice's cells."""
    g = n_side - 1
    xyz, conn = _lattice(dim, n_side)
    cen = torch.from_numpy(xyz).to(DEV)[torch.from_numpy(conn).to(DEV).long()].mean(1)
    c = torch.floor(cen * g).clamp(0, g - 1).long()
    flat = sum(c[:, k] * g ** k for k in range(dim))
    n = torch.zeros(g ** dim, dtype=torch.float64, device=DEV).index_add_(
        0, flat, torch.ones_like(cen[:, 0]))
    total = torch.zeros((g ** dim, dim), dtype=torch.float64, device=DEV).index_add_(0, flat, cen)
    return total / n[:, None], n > 0


def _features(dim, n_side, xp, pooled):
    g, W = n_side - 1, 9 if dim == 2 else 7
    mean, has = pooled
    c0 = torch.floor(xp * g).clamp(0, g - 1).long()
    r = torch.arange(W, device=DEV) - W // 2
    off = torch.stack(torch.meshgrid(*([r] * dim), indexing="ij")[::-1], dim=-1)
    cc = c0.reshape((-1,) + (1,) * dim + (dim,)) + off
    inside = ((cc >= 0) & (cc < g)).all(-1)
    flat = sum(cc[..., k].clamp(0, g - 1) * g ** k for k in range(dim))
    use = (inside & has[flat])[..., None]
    pt = torch.where(use, mean[flat], (cc.double() + 0.5) / g)
    win = (pt - xp.reshape((-1,) + (1,) * dim + (dim,))) * g
    return win.movedim(-1, 1), xp * g - (c0.double() + 0.5)


def _flat(grads):
    return torch.cat([t.reshape(-1) for t in grads])


def exact(case, seed):
    kind, dim = case["kind"], case["dim"]
    if kind == "predict":
        stride, n = case["stride"], case["n_side"]
        A, b = _linear_flow(dim, seed)
        g = (n - 1) // stride
        x = torch.from_numpy(_lattice(dim, n)[0]).to(DEV)
        u = x @ torch.from_numpy(A.T.copy()).to(DEV) + torch.from_numpy(b).to(DEV)
        s = stride / (n - 1)
        at = (torch.arange(g, dtype=torch.float64, device=DEV) + 0.5) * s
        pts = torch.stack(torch.meshgrid(*([at] * dim), indexing="ij")[::-1], dim=-1)
        U = pts @ torch.from_numpy(A.T.copy()).to(DEV) + torch.from_numpy(b).to(DEV)
        U = U * (_dt(u, n, 8.0) / s)
        R = 4 if dim == 2 else 3
        U = torch.nn.functional.pad(U.movedim(-1, 0)[None], (R, R) * dim)
        layers = _layers(_displacement_weights(dim), _predictor_layers(dim))
        return _predictor(U, layers).reshape(-1, dim)
    if kind == "grad":
        win, tgt = _windows(dim, case["batch"], seed)
        layers = _layers(_initial(_predictor_layers(dim), 10 + dim), _predictor_layers(dim))
        leaf = [t.detach().requires_grad_() for wb in layers for t in wb]
        out = _predictor(win.double(), list(zip(leaf[::2], leaf[1::2])))
        loss = (out.reshape(-1, dim) - tgt.double()).square().mean()
        return _flat(torch.autograd.grad(loss, leaf)), loss.detach()
    if kind in ("classify", "classify-grad"):
        n_side = case["n_side"]
        layers = _layers(_initial(_classifier_layers(dim), 20 + dim), _classifier_layers(dim))
        pooled = _pooled_centroids(dim, n_side)
        n = case["n"] if kind == "classify" else case["batch"]
        xp, gen = _departures(dim, n_side, n, seed)
        if kind == "classify":
            part = 8192 if dim == 2 else 1024
            return torch.cat([_classifier(*_features(dim, n_side, xp[i:i + part], pooled), layers)
                              for i in range(0, n, part)])
        label = _labels(dim, n_side, xp, gen).long()
        leaf = [t.detach().requires_grad_() for wb in layers for t in wb]
        H = _classifier(*_features(dim, n_side, xp, pooled), list(zip(leaf[::2], leaf[1::2])))
        loss = torch.nn.functional.cross_entropy(H, label)
        return _flat(torch.autograd.grad(loss, leaf)), loss.detach()
    return None      # hosts, path lengths and statuses are whole numbers
