"""Performance cases of the winding-number library: what its users have it do.

``listed()`` gives the fixed cases, ``draw(rng)`` one more of the same ranges,
``prepare(case, seed)`` what a program holds before the call (a built mesh and
queries on the GPU), ``run(state)`` one pass through the public entry points,
``work(case)`` the bytes and operations no implementation can do without, and
``exact(case, seed)`` the outputs in 64 bits by plain torch, where that takes
seconds.  The meshes have the structure and the sizes of this repository's
workloads (open caps, displaced spheres with small holes, integer staircases,
random triangle soups, height fields, superquadrics, random Bezier patches);
they are generated on the GPU, so that making them is quick.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2605_01536_gb300 as gwn

DEV = "cuda"


def listed():
    return [
        # a point pick or a probe: a few queries on a small open part, where latency is all
        {"name": "query_cap_64", "op": "query", "mesh": "cap", "level": 3, "n": 64},
        # a scan with small holes, a medium and odd number of points (winding numbers and crossing counts)
        {"name": "query_soup6_50k", "op": "query", "mesh": "soup", "level": 6, "n": 50_001},
        # inside/outside labels of millions of points against a scan of 2.6M triangles with 48k holes: the headline
        {"name": "classify_soup8_2M", "op": "classify", "mesh": "soup", "level": 8, "n": 2_000_000},
        # degenerate input: integer staircase and height field, queries on vertices, edges and faces
        {"name": "classify_staircase_500k", "op": "classify", "mesh": "staircase", "level": 40, "n": 500_000},
        # voxelisation of a closed solid: labels of a 256^3 grid
        {"name": "grid_closed_256", "op": "grid", "mesh": "closed", "level": 7, "n": 256},
        # grad w near a scan, as a reconstruction or an optimiser asks for it
        {"name": "gradient_soup6_100k", "op": "gradient", "mesh": "soup", "level": 6, "n": 100_003},
        # the plain solid-angle sum, the baseline that results are checked against
        {"name": "direct_soup5_30k", "op": "direct", "mesh": "soup", "level": 5, "n": 30_000},
        # a collection of parts of uneven sizes in one launch
        {"name": "batch_24", "op": "batch", "mesh": "mixed", "level": 24, "n": 20_000},
        # the learned surrogate: inference over a cloud, and a training gradient (forward and backward)
        {"name": "surrogate_predict_1M", "op": "predict", "mesh": "cap", "level": 3, "n": 1_000_000},
        {"name": "surrogate_grad_64k", "op": "mlp_grad", "mesh": "cap", "level": 3, "n": 65_536},
        # voxelisation of a parametric surface: 100 random bicubic patches, 32^3 cells
        {"name": "param_grid_32", "op": "param_grid", "mesh": "bezier", "level": 100, "n": 32},
        # ingest and acceleration build of a new scan, its boundary and its first 1,000 answers
        {"name": "build_soup7", "op": "build", "mesh": "soup", "level": 7, "n": 0},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["query", "query", "classify", "classify", "grid", "gradient", "direct", "batch", "predict",
                     "mlp_grad", "param_grid", "param", "build"])
    if op in ("query", "classify", "gradient"):
        kind = rng.choice(["cap", "soup", "staircase", "field", "triangles"])
        level = {"cap": lambda: rng.randint(2, 6), "soup": lambda: rng.randint(4, 8),
                 "staircase": lambda: rng.randint(8, 40), "field": lambda: _log_uniform(rng, 8, 400),
                 "triangles": lambda: _log_uniform(rng, 100, 30_000)}[kind]()
        top = 1_000_000 if kind in ("cap", "soup") else 200_000
        return {"op": op, "mesh": kind, "level": level, "n": _log_uniform(rng, 50, top)}
    if op == "grid":
        kind = rng.choice(["closed", "soup", "field"])
        level = _log_uniform(rng, 8, 400) if kind == "field" else rng.randint(4, 7)
        return {"op": op, "mesh": kind, "level": level, "n": _log_uniform(rng, 9, 256 if kind == "closed" else 80)}
    if op == "direct":
        return {"op": op, "mesh": rng.choice(["cap", "soup"]), "level": rng.randint(3, 5), "n": _log_uniform(rng, 50, 60_000)}
    if op == "batch":
        return {"op": op, "mesh": "mixed", "level": rng.randint(2, 32), "n": _log_uniform(rng, 1_000, 20_000)}
    if op in ("predict", "mlp_grad"):
        return {"op": op, "mesh": "cap", "level": 3, "n": _log_uniform(rng, 100, 2_000_000 if op == "predict" else 200_000)}
    if op == "param_grid":
        return {"op": op, "mesh": "bezier", "level": _log_uniform(rng, 4, 150), "n": rng.randint(5, 34)}
    if op == "param":
        return {"op": op, "mesh": "bezier", "level": _log_uniform(rng, 4, 150), "n": _log_uniform(rng, 50, 30_000)}
    return {"op": op, "mesh": rng.choice(["soup", "closed"]), "level": rng.randint(3, 7), "n": 0}


# ------------------------------------------------------------------ meshes ----

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float64)


def _cross(a, b):
    return torch.linalg.cross(a, b, dim=-1)


def _icosphere(level):
    """Unit sphere of 20 * 4**level outward faces (float64 vertices, int64 faces)."""
    t = (1.0 + math.sqrt(5.0)) / 2.0
    V = torch.tensor([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t], [0, -1, -t], [0, 1, -t],
                      [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]], dtype=torch.float64, device=DEV)
    F = torch.tensor([[0, 11, 5], [0, 5, 1], [0, 1, 7], [0, 7, 10], [0, 10, 11], [1, 5, 9], [5, 11, 4], [11, 10, 2],
                      [10, 7, 6], [7, 1, 8], [3, 9, 4], [3, 4, 2], [3, 2, 6], [3, 6, 8], [3, 8, 9], [4, 9, 5],
                      [2, 4, 11], [6, 2, 10], [8, 6, 7], [9, 8, 1]], dtype=torch.int64, device=DEV)
    V = V / V.norm(dim=1, keepdim=True)
    for _ in range(level):
        nv = V.shape[0]
        e = torch.cat([F[:, [0, 1]], F[:, [1, 2]], F[:, [2, 0]]])
        uniq, inv = torch.unique(e.min(1).values * nv + e.max(1).values, return_inverse=True)
        mid = V[uniq // nv] + V[uniq % nv]
        V = torch.cat([V, mid / mid.norm(dim=1, keepdim=True)])
        ab, bc, ca = (nv + inv).chunk(3)
        a, b, c = F.unbind(1)
        F = torch.cat([torch.stack(s, 1) for s in ((a, ab, ca), (ab, b, bc), (ca, bc, c), (ab, bc, ca))])
    return V, F


def _rotation(g):
    Q, R = torch.linalg.qr(_randn(g, 3, 3))
    Q = Q * torch.sign(torch.diagonal(R))
    return Q if torch.det(Q) > 0 else -Q


def _grid_faces(n, m):
    i, j = torch.meshgrid(torch.arange(n - 1, device=DEV), torch.arange(m - 1, device=DEV), indexing="ij")
    a, b = (i * m + j).reshape(-1), ((i + 1) * m + j).reshape(-1)
    c, d = b + 1, a + 1
    return torch.cat([torch.stack([a, b, c], 1), torch.stack([a, c, d], 1)])


def _soup(level, hole, g):
    """Displaced sphere and a shifted, intersecting copy; a share ``hole`` of the faces is missing
    (the same faces for every seed, so that the boundary's size is the case's)."""
    V, F = _icosphere(level)
    phase = 2.0 * math.pi * _rand(g, 3)
    V = V * (1.0 + 0.05 * torch.sin(5.0 * V + phase).prod(1, keepdim=True))
    F = torch.cat([F, F + V.shape[0]])
    V = torch.cat([V, V + torch.tensor([0.3, 0.0, 0.0], dtype=torch.float64, device=DEV)])
    return V, F[_rand(_generator(level), F.shape[0]) >= hole] if hole > 0 else F


def _cap(level, g):
    """Sphere without the faces above z = 0.8: one open loop; turned a little about z for each seed."""
    V, F = _icosphere(level)
    a = float(_rand(g, 1)) * 2.0 * math.pi
    R = torch.tensor([[math.cos(a), -math.sin(a), 0.0], [math.sin(a), math.cos(a), 0.0], [0.0, 0.0, 1.0]],
                     dtype=torch.float64, device=DEV)
    return V @ R.T, F[V[F].mean(1)[:, 2] <= 0.8]


def _triangles(nt, g):
    """Unwelded random triangles in the unit cube, edges up to a fifth of it."""
    p, L = _rand(g, nt, 3), 0.01 + 0.19 * _rand(g, nt, 1)
    d = _randn(g, 2, nt, 3)
    d = d / d.norm(dim=2, keepdim=True)
    return torch.stack([p, p + L * d[0], p + L * d[1]], 1).reshape(-1, 3), torch.arange(3 * nt, device=DEV).reshape(-1, 3)


def _field(n, g):
    """Open rough height field of n x n vertices, turned in space."""
    x = torch.linspace(0, 1, n, device=DEV, dtype=torch.float64)
    X, Y = torch.meshgrid(x, x, indexing="ij")
    V = torch.stack([X, Y, 0.1 * _randn(g, n, n)], -1).reshape(-1, 3)
    return V @ _rotation(g).T, _grid_faces(n, n)


def _superquadric(nt, g):
    """Closed superquadric on a latitude/longitude grid, welded, outward."""
    e1, e2 = (0.3 + 2.7 * _rand(g, 2)).tolist()
    nu = max(3, int(round(math.sqrt(nt / 2.0))))
    nr = max(1, int(round(nt / (2.0 * nu))) - 1)
    eta = -math.pi / 2 + math.pi * torch.arange(1, nr + 1, device=DEV, dtype=torch.float64)[:, None] / (nr + 1)
    om = 2.0 * math.pi * torch.arange(nu, device=DEV, dtype=torch.float64)[None] / nu
    p = lambda c, e: torch.sign(c) * c.abs() ** e
    ring = torch.stack([p(eta.cos(), e1) * p(om.cos(), e2), p(eta.cos(), e1) * p(om.sin(), e2),
                        p(eta.sin(), e1).expand(nr, nu)], -1).reshape(-1, 3)
    V = torch.cat([ring, torch.tensor([[0.0, 0.0, -1.0], [0.0, 0.0, 1.0]], dtype=torch.float64, device=DEV)])
    c = torch.arange(nu, device=DEV)
    d = (c + 1) % nu
    F = [torch.stack([torch.full_like(c, nr * nu), d, c], 1),
         torch.stack([(nr - 1) * nu + c, (nr - 1) * nu + d, torch.full_like(c, nr * nu + 1)], 1)]
    if nr > 1:
        r = (torch.arange(nr - 1, device=DEV) * nu)[:, None]
        q = [(r + c).reshape(-1), (r + d).reshape(-1), (r + nu + d).reshape(-1), (r + nu + c).reshape(-1)]
        F += [torch.stack([q[0], q[1], q[2]], 1), torch.stack([q[0], q[2], q[3]], 1)]
    V = (V * (0.5 + 1.5 * _rand(g, 3))) @ _rotation(g).T + 2.0 * _rand(g, 3) - 1.0
    return V, torch.cat(F)


def _staircase(radius, g):
    """Closed surface of the unit voxels inside a sphere, and an open integer height field above it."""
    R = radius + 1
    ax = torch.arange(-R, R, device=DEV)
    ctr = (ax + 0.5) ** 2
    inside = ctr[:, None, None] + ctr[None, :, None] + ctr[None, None, :] < radius * radius
    corners = {0: [(0, 0, 0), (0, 0, 1), (0, 1, 1), (0, 1, 0)], 1: [(0, 0, 0), (1, 0, 0), (1, 0, 1), (0, 0, 1)],
               2: [(0, 0, 0), (0, 1, 0), (1, 1, 0), (1, 0, 0)]}
    quads = []
    for axis in range(3):
        for side in (0, 1):
            face = inside & ~torch.roll(inside, 1 - 2 * side, axis)
            base = face.nonzero() - R
            off = torch.tensor(corners[axis], device=DEV)
            if side:
                off = off.flip(0)
                off[:, axis] = 1
            quads.append(base[:, None, :] + off[None])
    P = torch.cat(quads)
    w = 4 * R
    key, inv = torch.unique(((P[..., 0] + w) * 2 * w + P[..., 1] + w) * 2 * w + P[..., 2] + w, return_inverse=True)
    V = torch.stack([key // (4 * w * w) - w, key // (2 * w) % (2 * w) - w, key % (2 * w) - w], 1).double()
    F = torch.cat([inv[:, [0, 1, 2]], inv[:, [0, 2, 3]]])
    n = 5 * radius
    h = radius + 5 + torch.randint(-3, 4, (n, n), generator=g, device=DEV)
    i, j = torch.meshgrid(torch.arange(n, device=DEV), torch.arange(n, device=DEV), indexing="ij")
    patch = torch.stack([i - n // 2, j - n // 2, h], -1).reshape(-1, 3).double()
    return torch.cat([V, patch]), torch.cat([F, _grid_faces(n, n) + V.shape[0]]), F.shape[0]


def _mesh(kind, level, g):
    if kind == "cap":
        V, F = _cap(level, g)
    elif kind == "soup":
        V, F = _soup(level, 0.02, g)
    elif kind == "closed":
        V, F = _soup(level, 0.0, g)
    elif kind == "field":
        V, F = _field(level, g)
    elif kind == "triangles":
        V, F = _triangles(level, g)
    else:
        V, F, _ = _staircase(level, g)
    return V.float(), F.int()


def _bounds(V, pad):
    lo, hi = V.double().min(0).values, V.double().max(0).values
    return lo - pad * (hi - lo), hi + pad * (hi - lo)


def _queries(V, F, n, g):
    """Half uniform in the padded box, half within about 1e-3 of the surface."""
    V = V.double()
    lo, hi = _bounds(V, 0.1)
    k = n - n // 2
    far = lo + _rand(g, k, 3) * (hi - lo)
    P = V[F.long()]
    area = _cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]).norm(dim=1).cumsum(0)
    t = torch.searchsorted(area, _rand(g, n // 2) * area[-1], right=True).clamp(max=F.shape[0] - 1)
    s, r = _rand(g, n // 2, 1).sqrt(), _rand(g, n // 2, 1)
    near = (1 - s) * P[t, 0] + s * (1 - r) * P[t, 1] + s * r * P[t, 2] + 1e-3 * _randn(g, n // 2, 3)
    return torch.cat([far, near]).float().contiguous()


def _degenerate_queries(V, F, n, g):
    """Queries exactly on vertices, edge midpoints, points of faces and grid points of an integer mesh."""
    V, F = V.double(), F.long()
    k = (n + 3) // 4
    pick = lambda m: torch.randint(0, m, (k,), generator=g, device=DEV)
    t, e = pick(F.shape[0]), pick(3)
    P = V[F[pick(F.shape[0])]]
    u = torch.randint(0, 9, (k, 1), generator=g, device=DEV).double() / 8
    v = torch.randint(0, 9, (k, 1), generator=g, device=DEV).double() / 8 * (1 - u)
    lo, hi = V.min(0).values - 1, V.max(0).values + 1
    return torch.cat([V[pick(V.shape[0])], 0.5 * (V[F[t, e]] + V[F[t, (e + 1) % 3]]),
                      P[:, 0] + u * (P[:, 1] - P[:, 0]) + v * (P[:, 2] - P[:, 0]),
                      torch.floor(lo + _rand(g, k, 3) * (hi - lo + 1))])[:n].float().contiguous()


def _axes(V, n):
    """Cell centres of about n per axis (not the same number on each) over the padded box."""
    lo, hi = (x.tolist() for x in _bounds(V, 0.1))
    sizes = (n, max(1, n - n // 16), n)
    return [np.asarray([lo[d] + (i + 0.5) * (hi[d] - lo[d]) / m for i in range(m)], np.float32) for d, m in enumerate(sizes)]


def _collection(case, g):
    """Meshes of uneven sizes, cycling closed superquadric, open height field, random triangles."""
    out = []
    for i in range(case["level"]):
        nt = int(round(100 * 500 ** (0.618034 * (i + 1) % 1)))           # 100 to 50,000 triangles
        nq = int(round(case["n"] * 100 ** (0.754878 * (i + 1) % 1 - 0.5)))   # a tenth to ten times n queries
        if i % 3 == 0:
            V, F = _superquadric(nt, g)
        elif i % 3 == 1:
            V, F = _field(max(2, int(round(math.sqrt(nt / 2.0))) + 1), g)
        else:
            V, F = _triangles(nt, g)
        V, F = V.float(), F.int()
        out.append((V, F, _queries(V, F, max(nq, 2), g)))
    return out


def _network(g):
    """Random weights of the surrogate network, in its documented order, scaled so that the layers keep their size."""
    parts = []
    for fan, shape in ((99, (64, 128)), (64, (64, 64)), (64, (64, 64)), (64, (64, 64)), (64, (1, 64))):
        parts += [(_randn(g, *shape) * math.sqrt(2.0 / fan)).reshape(-1), 0.1 * _randn(g, shape[0])]
    return torch.cat(parts).float().cpu().numpy()


def _inputs(case, seed):
    g = _generator(seed)
    op = case["op"]
    if op == "batch":
        return {"parts": _collection(case, g)}
    if op in ("param", "param_grid"):
        P = _rand(g, case["level"], 4, 4, 3).float()
        lo, hi = _bounds(P.reshape(-1, 3), 0.1)
        x = {"patches": P.cpu().numpy(), "axes": _axes(P.reshape(-1, 3), case["n"])}
        x["q"] = (lo + _rand(g, case["n"], 3) * (hi - lo)).float().contiguous()
        return x
    V, F = _mesh(case["mesh"], case["level"], g)
    x = {"V": V, "F": F}
    if op == "grid":
        x["axes"] = _axes(V, case["n"])
    elif op == "build":
        x["q"] = _queries(V, F, 1_000, g)
        x["V"], x["F"] = V.cpu().numpy(), F.cpu().numpy()
    elif case["mesh"] == "staircase":
        x["q"] = _degenerate_queries(V, F, case["n"], g)
    else:
        x["q"] = _queries(V, F, case["n"], g)
    if op in ("predict", "mlp_grad"):
        x["params"] = _network(g)
        x["box"] = np.asarray([-1.5, -1.5, -1.5, 1.5, 1.5, 1.5], np.float32)
        x["targets"] = _rand(g, case["n"]).float()
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    op = case["op"]
    x["op"] = op
    if op == "batch":
        x["meshes"] = [gwn.Mesh(V, F) for V, F, _ in x["parts"]]
        x["batch"] = gwn.Batch(x["meshes"], [len(q) for _, _, q in x["parts"]])
        x["q"] = torch.cat([q for _, _, q in x["parts"]]).contiguous()
    elif op in ("param", "param_grid"):
        x["surface"] = gwn.ParamSurface(x["patches"])
    elif op != "build":
        x["m"] = gwn.Mesh(x["V"], x["F"], build=op != "direct")
        if "params" in x:
            x["m"].set_surrogate_params(x["params"], x["box"])
    return x


def run(state):
    op = state["op"]
    if op == "query":
        return state["m"].query(state["q"])
    if op == "classify":
        return state["m"].classify(state["q"], want_w=True)
    if op == "grid":
        return state["m"].classify_grid(*state["axes"], want_w=True)
    if op == "gradient":
        return state["m"].gradient(state["q"])
    if op == "direct":
        return state["m"].direct(state["q"])
    if op == "batch":
        return state["batch"].run(state["q"])
    if op == "predict":
        return state["m"].surrogate_predict(state["q"])
    if op == "mlp_grad":
        return state["m"].surrogate_grad(state["q"], state["targets"])
    if op == "param":
        return state["surface"].query(state["q"])
    if op == "param_grid":
        return state["surface"].query_grid(*state["axes"])
    m = gwn.Mesh(state["V"], state["F"])
    out = (m.boundary_edges(), m.boundary_points()) + m.query(state["q"])
    m.close()
    return out


# -------------------------------------------------------------- accounting ----

def _counts(case):
    """(triangles, boundary edges) of the case's mesh, near enough for accounting."""
    k, L = case["mesh"], case["level"]
    if k in ("soup", "closed"):
        nt = 40 * 4 ** L
        return (0.98 * nt, 0.06 * nt) if k == "soup" else (nt, 0)
    if k == "cap":
        return 18 * 4 ** L, 4.5 * 2 ** L
    if k == "field":
        return 2 * (L - 1) ** 2, 4 * (L - 1)
    if k == "triangles":
        return L, 3 * L
    return 37.7 * L * L + 50 * L * L, 20 * L


def work(case):
    """Inputs read once and outputs written once.  Operations: the direct sum visits every
    triangle (70 each); the boundary sum is charged one term (56 operations) for each level of a
    hierarchy over the boundary, the least a far-field method can do; the network its products;
    the parametric integrals one 15-point panel per curve."""
    op, n = case["op"], case["n"]
    if op == "batch":
        q = 1.8 * n * case["level"]   # mean of the uneven query counts
        return {"bytes": 20.0 * q + 54.0 * 8_000 * case["level"], "flops": q * 56 * 10}
    if op in ("param", "param_grid"):
        cells = n if op == "param" else len(range(n)) ** 2 * max(1, n - n // 16)
        return {"bytes": 192.0 * case["level"] + (20.0 if op == "param" else 8.0) * cells,
                "flops": cells * 4.0 * case["level"] * 1122}
    nt, nb = _counts(case)
    mesh = 12.0 * nt + 6.0 * nt   # faces, and half as many vertices
    if op == "build":
        return {"bytes": mesh + 36.0 * nb, "flops": 60.0 * nt}
    if op in ("predict", "mlp_grad"):
        f = 2.0 * (128 * 64 + 3 * 64 * 64 + 64) * n
        return {"bytes": 16.0 * n + 83_204, "flops": f if op == "predict" else 3 * f}
    terms = 56.0 * math.log2(nb + 2) if nb else 0.0
    if op == "grid":
        cells = n * n * max(1, n - n // 16)
        return {"bytes": mesh + 5.0 * cells, "flops": cells * (1 + terms)}
    if op == "direct":
        return {"bytes": mesh + 16.0 * n, "flops": 70.0 * nt * n}
    out = {"query": 8, "classify": 5, "gradient": 12}[op]
    return {"bytes": mesh + (12.0 + out) * n, "flops": n * (30 + terms)}


# ---------------------------------------------------------- 64-bit results ----

def _solid_angles(q, V, F):
    """Sum of the triangles' signed solid angles over 4 pi, in 64 bits."""
    P, q = V.double()[F.long()], q.double()
    out = torch.empty(len(q), dtype=torch.float64, device=DEV)
    step = max(1, 40_000_000 // max(1, len(P)))
    for i in range(0, len(q), step):
        a, b, c = ((P[None, :, k] - q[i:i + step, None]).unbind(-1) for k in range(3))
        norm = lambda u: (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]).sqrt()
        dot = lambda u, v: u[0] * v[0] + u[1] * v[1] + u[2] * v[2]
        la, lb, lc = norm(a), norm(b), norm(c)
        det = (a[0] * (b[1] * c[2] - b[2] * c[1]) + a[1] * (b[2] * c[0] - b[0] * c[2])
               + a[2] * (b[0] * c[1] - b[1] * c[0]))
        den = la * lb * lc + dot(a, b) * lc + dot(a, c) * lb + dot(b, c) * la
        out[i:i + step] = torch.atan2(det, den).sum(1)
    return out / (2.0 * math.pi)


def _boundary(F, nv):
    """Directed edges that no opposite edge cancels."""
    F = F.long()
    e = torch.cat([F[:, [0, 1]], F[:, [1, 2]], F[:, [2, 0]]])
    key, inv = torch.unique(e.min(1).values * nv + e.max(1).values, return_inverse=True)
    net = torch.zeros(len(key), dtype=torch.int64, device=DEV)
    net.scatter_add_(0, inv, torch.where(e[:, 0] < e[:, 1], 1, -1))
    at = net.nonzero()[:, 0]
    lo, hi = key[at] // nv, key[at] % nv
    m = net[at]
    E = torch.where((m > 0)[:, None], torch.stack([lo, hi], 1), torch.stack([hi, lo], 1))
    return E.repeat_interleave(m.abs(), 0)


def _gradient(q, V, F):
    """Gradient of the solid angle of the boundary curve over 4 pi: the sum over its segments of
    (a x b) (|a| + |b|) / (|a| |b| (|a| |b| + a.b)), a and b from the query."""
    E, q = _boundary(F, len(V)), q.double()
    A, B = V.double()[E[:, 0]], V.double()[E[:, 1]]
    out = torch.zeros(len(q), 3, dtype=torch.float64, device=DEV)
    step = max(1, 20_000_000 // max(1, len(E)))
    for i in range(0, len(q), step):
        a, b = A[None] - q[i:i + step, None], B[None] - q[i:i + step, None]
        la, lb = a.norm(dim=2), b.norm(dim=2)
        f = (la + lb) / (la * lb * (la * lb + (a * b).sum(2)))
        out[i:i + step] = (_cross(a, b) * f[..., None]).sum(1)
    return out / (4.0 * math.pi)


def _features(q, box):
    lo, hi = (torch.as_tensor(box[s], dtype=torch.float64, device=DEV) for s in (slice(0, 3), slice(3, 6)))
    x = 2.0 * (q.double() - lo) / (hi - lo) - 1.0
    s = math.pi * 2.0 ** (7.0 * torch.arange(16, dtype=torch.float64, device=DEV) / 15.0)
    a = s[None, :, None] * x[:, None, :]
    f = torch.stack([a.sin(), a.cos()], -1).reshape(len(q), 96)
    return torch.cat([x, f, torch.zeros(len(q), 29, dtype=torch.float64, device=DEV)], 1)


def _forward(p, f):
    o, h = 0, f
    for rows, cols in ((64, 128), (64, 64), (64, 64), (64, 64), (1, 64)):
        W = p[o:o + rows * cols].reshape(rows, cols)
        b = p[o + rows * cols:o + rows * cols + rows]
        o += rows * cols + rows
        h = h @ W.T + b
        h = h.relu() if rows > 1 else h
    return h[:, 0]


def exact(case, seed):
    op = case["op"]
    if op in ("param", "param_grid"):
        return None
    x = _inputs(case, seed)
    if op == "batch":
        if sum(len(F) * len(q) for _, F, q in x["parts"]) > 1.5e10:
            return None
        return torch.cat([_solid_angles(q, V, F) for V, F, q in x["parts"]]), None
    if op in ("predict", "mlp_grad"):
        p = torch.as_tensor(x["params"], dtype=torch.float64, device=DEV).requires_grad_(op == "mlp_grad")
        if op == "predict":
            return torch.cat([_forward(p, _features(q, x["box"])) for q in x["q"].split(100_000)])
        if case["n"] > 200_000:
            return None
        loss = (_forward(p, _features(x["q"], x["box"])) - x["targets"].double()).square().mean()
        loss.backward()
        return p.grad, loss.detach()
    if case["mesh"] == "staircase":   # queries on the surface and on its boundary: no solid angle there
        return None
    V, F = (torch.as_tensor(x[k], device=DEV) for k in "VF")
    if op == "gradient":
        return _gradient(x["q"], V, F) if len(x["q"]) * len(_boundary(F, len(V))) < 1.5e10 else None
    if op == "grid":
        a = [torch.as_tensor(v, device=DEV) for v in x["axes"]]
        Z, Y, X = torch.meshgrid(a[2], a[1], a[0], indexing="ij")
        if X.numel() * len(F) > 1.5e10:
            return None
        return None, _solid_angles(torch.stack([X, Y, Z], -1).reshape(-1, 3), V, F).reshape(X.shape)
    if len(x["q"]) * len(F) > 1.5e10:
        return None
    w = _solid_angles(x["q"], V, F)
    return {"query": (w, None), "classify": (None, w), "direct": w, "build": (None, None, w, None)}[op]
