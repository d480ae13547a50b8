"""Measured workloads of the walk-on-boundary library.

Each case is one call (or one short sequence of calls) that a program using
the library makes, over the range of sizes it is used at: the double-layer
solve from a few thousand walks to a dense slice, value and gradient, many
problems in one batch, the single-layer and direct-integral Neumann / Robin
walks, mixed conditions with resampling, the forward paths, the learned
control variate with its network and its training step, and the set-up of a
new boundary.  ``exact`` restates what the calls compute in plain torch,
64 bits and brute force over every triangle (same counter-based streams).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2305_04403_gb300 as wob
from paper_2305_04403_gb300 import inputs as I

# Brute-force line x triangle pairs that exact() takes on (a few seconds).
MAX_PAIRS = 1.5e10
X_FAR = (0.0, 0.0, 5.0)      # point source above the boundary
X_SIDE = (3.0, 0.0, 0.0)     # point source beside it
X_TUBE = (1.0, 0.0, 0.0)     # point source inside the torus tube


def listed():
    return [
        # the smallest solve: a few hundred probes on a coarse ball with
        # vertex data, as an interactive tool or a test makes it
        dict(name="dl_small", path="dl", mesh="ico", size=3, side=1, data="p1", queries=256,
             walks=64, length=4),
        # the headline path: a slice through the level-6 star
        dict(name="dl_star_slice", path="dl", mesh="star", size=6, side=1, data="point",
             queries=0, grid=128, walks=512, length=16),
        # value and gradient together (field lines, normal derivatives)
        dict(name="grad_spiky", path="grad", mesh="spiky", size=5, side=1, data="point",
             queries=4096, walks=128, length=8),
        # many small independent problems in one graph replay
        dict(name="batch_24", path="batch", problems=24, tri_hi=20000, query_hi=2048, walks=128),
        # exterior Robin, single layer, area sampling
        dict(name="sl_robin", path="sl", mesh="torus", size=100, side=-1, alpha=2.0, data="point",
             kind=wob.ROBIN_SL, ris=0, queries=32768, walks=256, length=24),
        # mixed Dirichlet / Neumann / Robin parts with 16 candidates a step
        dict(name="mixed_ris", path="sl", mesh="torus", size=100, side=1, alpha=1.0, data="point",
             kind=wob.MIXED_SL, ris=16, queries=8192, walks=128, length=4),
        # interior Neumann through the direct integral equation, half of the
        # queries on the boundary
        dict(name="nd_torus", path="nd", mesh="torus", size=100, side=1, data="point",
             queries=8192, walks=128, length=24),
        # forward paths from sparse data, connected to every query
        dict(name="fwd_bump", path="fwd", mesh="torus", size=40, side=1, data="bump",
             paths=16384, queries=32768, length=24),
        # residual walks of the learned control variate
        dict(name="cv_solve", path="cv", mesh="ico", size=3, side=1, data="poly", queries=8192,
             walks=64, length=2),
        # the control variate's network on a million points
        dict(name="mlp_forward", path="mlp", points=1 << 20),
        # one training step of it
        dict(name="mlp_train", path="train", points=4096),
        # a new boundary: mesh, tree and a short first solve
        dict(name="new_boundary", path="setup", mesh="torus", size=100, side=1, data="point",
             queries=1024, walks=16, length=4),
    ]


def _between(rng, lo, hi):
    """A whole number spread over the logarithm of [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["dl", "dl", "grad", "batch", "sl", "sl", "nd", "fwd", "cv", "mlp", "train",
                       "setup"])
    c = dict(path=path)
    if path in ("dl", "grad", "setup"):
        c["mesh"] = rng.choice(["ico", "star", "spiky", "torus"])
        c["size"] = _between(rng, 16, 100) if c["mesh"] == "torus" else rng.randint(3, 6)
        c["side"] = rng.choice([1, 1, -1])
        c["data"] = rng.choice(["p1", "point", "poly"] if c["side"] == 1 else ["p1", "point"])
        c["length"] = rng.randint(1, 16)
        c["queries"] = _between(rng, 100, 6000 if path == "dl" else 2500)
        c["walks"] = _between(rng, 20, 300 if path == "dl" else 120)
    elif path == "batch":
        c.update(problems=rng.randint(3, 24), tri_hi=_between(rng, 1000, 20000),
                 query_hi=_between(rng, 100, 2000), walks=_between(rng, 33, 128))
    elif path == "sl":
        kind = rng.choice([wob.NEUMANN_SL, wob.ROBIN_SL, wob.MIXED_SL])
        ris = rng.choice([0, 0, 4, 16])
        c.update(mesh="torus", size=_between(rng, 16, 100), side=rng.choice([1, -1]), kind=kind,
                 alpha=0.0 if kind == wob.NEUMANN_SL else rng.choice([0.5, 1.0, 2.0]), ris=ris,
                 data=rng.choice(["point", "point", "p1"]) if kind == wob.NEUMANN_SL else "point",
                 queries=_between(rng, 500, 20000), walks=_between(rng, 30, 200 if not ris else 60),
                 length=rng.randint(2, 24 if not ris else 6))
    elif path == "nd":
        c.update(mesh="torus", size=_between(rng, 16, 100), side=1,
                 data=rng.choice(["point", "p1"]), queries=_between(rng, 300, 8000),
                 walks=_between(rng, 20, 120), length=rng.randint(2, 24))
    elif path == "fwd":
        c.update(mesh="torus", size=_between(rng, 16, 100), side=1, data="bump",
                 paths=_between(rng, 500, 16000), queries=_between(rng, 300, 60000),
                 length=rng.randint(2, 24))
    elif path == "cv":
        c.update(mesh="ico", size=rng.choice([2, 3, 3]), side=1, data="poly",
                 queries=_between(rng, 300, 8000), walks=_between(rng, 8, 64),
                 length=rng.randint(1, 3))
    elif path == "mlp":
        c["points"] = _between(rng, 1000, 2000000)
    else:
        c["points"] = _between(rng, 300, 40000)
    return c


# ---------------------------------------------------------------- inputs
def _mesh(c):
    s = c["size"]
    if c["mesh"] == "ico":
        return (*I.icosphere(s), None)
    if c["mesh"] == "star":
        return I.star_mesh(s)
    if c["mesh"] == "spiky":
        return I.star_mesh(s, seed=3, decay=0.5)
    return I.displaced_torus(5 * s, 2 * s)


def _queries(c, shape, seed):
    """Probe points of the case: float32 (Q, 3)."""
    n, inside = c["queries"], c["side"] == 1
    if c["mesh"] == "torus":
        return I.torus_queries(shape, n, inside, seed)
    if c.get("grid"):  # a slice, moved a little with the seed
        q = I.star_slice_queries(shape, c["grid"], margin=3e-2)
        return q + np.random.default_rng(seed).uniform(-5e-3, 5e-3, 3).astype(np.float32)
    rng = np.random.default_rng(seed)
    g = rng.standard_normal((n, 3))
    g /= np.linalg.norm(g, axis=1, keepdims=True)
    r = shape.radius(g) if shape is not None else np.ones(n)
    r = r * (0.05 + 0.85 * rng.random(n)) if inside else r * (1.1 + rng.random(n))
    return (g * r[:, None]).astype(np.float32)


def _data(c, v, f, seed):
    """Boundary data as the problem's arguments."""
    inside = c["side"] == 1
    if c["data"] == "p1":
        return dict(data_mode=wob.DATA_VERTEX_P1,
                    vertex_data=torch.from_numpy(I.poly_eval(I.POLY_CONFIG1, v).astype(np.float32)).cuda())
    if c["data"] == "bump":
        return dict(data_mode=wob.DATA_VERTEX_P1,
                    vertex_data=torch.from_numpy(I.bump_data(v, f, seed=seed % 1000)).cuda())
    if c["data"] == "poly":
        return dict(data_mode=wob.DATA_POLY, poly=I.POLY_CONFIG1)
    if inside:
        return dict(data_mode=wob.DATA_POINT, x0=X_SIDE if c["path"] in ("dl", "grad", "setup") else X_FAR)
    return dict(data_mode=wob.DATA_POINT, x0=X_TUBE if c["mesh"] == "torus" else (0.0, 0.0, 0.1))


KINDS = {"dl": wob.DIRICHLET_DL, "grad": wob.DIRICHLET_DL, "setup": wob.DIRICHLET_DL,
         "cv": wob.DIRICHLET_DL, "nd": wob.NEUMANN_DIRECT, "fwd": wob.NEUMANN_SL}


def _args(c, v, f, seed):
    """Every argument of the case's problem but its tree."""
    a = dict(kind=c.get("kind", KINDS.get(c["path"])), side=c["side"], alpha=c.get("alpha", 0.0),
             ris=c.get("ris", 0), **_data(c, v, f, seed))
    if a["kind"] == wob.MIXED_SL:
        bc = np.random.default_rng(seed).integers(0, 3, len(f)).astype(np.uint8)
        a.update(bc_type=torch.from_numpy(bc).cuda(), k_mix=1.5 if c["side"] == 1 else 4.0, p_k=2.0 / 3.0)
    return a


def _scene(c, seed):
    """Host mesh, problem arguments and queries (with the triangle of each,
    -1 off the boundary) of a single-mesh case."""
    v, f, shape = _mesh(c)
    q = _queries(c, shape, seed)
    prim = None
    if c["path"] == "nd":  # every second query lies on the boundary
        b, p = I.boundary_points(v, f, len(q), seed)
        prim = np.where(np.arange(len(q)) % 2 == 0, p, -1).astype(np.int32)
        q = np.where(prim[:, None] >= 0, b, q).astype(np.float32)
    return v, f, _args(c, v, f, seed), q, prim


def _batch_items(c, seed):
    """The seeded batch of problems, its probe points moved with the seed
    (they keep their margin to the boundary)."""
    items = I.batch_workload(c["problems"], (500, c["tri_hi"]), (64, c["query_hi"]))
    rng = np.random.default_rng(seed)
    for it in items:
        it.queries = it.queries + rng.uniform(-5e-3, 5e-3, it.queries.shape).astype(np.float32)
    return items


def _sphere_points(n, seed):
    g = torch.Generator("cuda").manual_seed(seed)
    x = torch.randn(n, 3, device="cuda", generator=g)
    return x / x.norm(dim=1, keepdim=True), g


def _train_state(c, seed):
    """A network in the middle of its training: weights, Adam's moments, a
    minibatch of boundary points and their density targets."""
    x, g = _sphere_points(c["points"], seed)
    p = wob.mlp_init(seed)
    m = 1e-3 * torch.randn(p.shape, device="cuda", generator=g)
    v = 1e-6 + m * m
    t = 2 * (x[:, 0] ** 2 - x[:, 1] ** 2 + 0.5 * x[:, 2]) + 0.3 * torch.randn(
        c["points"], device="cuda", generator=g)
    return p, m, v, x, t


# ---------------------------------------------------------------- passes
def prepare(c, seed):
    path = c["path"]
    if path == "mlp":
        x, _ = _sphere_points(c["points"], seed)
        return dict(path=path, x=x, params=wob.mlp_init(seed))
    if path == "train":
        p, m, v, x, t = _train_state(c, seed)
        return dict(path=path, params=p, m=m, v=v, x=x, t=t, grad=torch.empty_like(p),
                    loss=torch.empty(1, device="cuda"))
    if path == "batch":
        items = _batch_items(c, seed)
        probs = []
        for i, it in enumerate(items):
            bvh = wob.build_bvh(wob.build_mesh(it.verts, it.tris))
            probs.append(wob.Problem(bvh, kind=wob.DIRICHLET_DL, side=1, data_mode=wob.DATA_POINT,
                                     x0=X_SIDE, problem=i))
        b = wob.Batch(probs, [it.queries for it in items], c["walks"], [it.max_len for it in items],
                      tile_rounds=1, order=1)
        return dict(path=path, batch=b, seed=seed)
    v, f, args, q, prim = _scene(c, seed)
    s = dict(path=path, q=torch.from_numpy(q).cuda(), seed=seed, length=c["length"],
             prim=None if prim is None else torch.from_numpy(prim).cuda())
    vd, fd = torch.from_numpy(v).cuda(), torch.from_numpy(f).cuda()
    s.update({k: c[k] for k in ("walks", "paths") if k in c})
    if path == "setup":
        return dict(s, verts=vd, tris=fd, args=args)
    mesh = wob.build_mesh(vd, fd)
    s["prob"] = wob.Problem(wob.build_bvh(mesh), **args)
    if path == "cv":
        s["cv"] = wob.ControlVariate(mesh)
        s["params"] = wob.mlp_init(seed)
        s["cv"].set_network(s["params"])
        s["sums"] = torch.empty(2, len(q), dtype=torch.float64, device="cuda")
        s["dnt"] = torch.empty(len(q), device="cuda")
    return s


def run(s):
    path = s["path"]
    if path in ("dl", "sl", "nd"):
        return wob.solve(s["prob"], s["q"], s["walks"], s["length"], seed=s["seed"],
                         query_prim=s["prim"])
    if path == "grad":
        return wob.solve_grad(s["prob"], s["q"], s["walks"], s["length"], seed=s["seed"])
    if path == "batch":
        return s["batch"].run(s["seed"])
    if path == "fwd":
        return wob.solve_forward(s["prob"], s["q"], s["paths"], s["length"], seed=s["seed"])
    if path == "cv":
        s["sums"].zero_()
        s["cv"].solve_range(s["prob"], s["params"], s["q"], 0, s["walks"], s["length"],
                            s["sums"][0], s["sums"][1], seed=s["seed"], dnt=s["dnt"])
        return s["sums"], s["dnt"]
    if path == "mlp":
        return wob.mlp_forward(s["params"], s["x"])
    if path == "train":
        wob.mlp_train_step(s["params"], s["m"], s["v"], s["x"], s["t"], 1e-3, 1000, grad=s["grad"],
                           loss=s["loss"])
        return s["params"], s["m"], s["v"], s["grad"], s["loss"]
    mesh = wob.build_mesh(s["verts"], s["tris"])  # setup: a boundary seen for the first time
    prob = wob.Problem(wob.build_bvh(mesh), **s["args"])
    return wob.solve(prob, s["q"], s["walks"], s["length"], seed=s["seed"])


def _tris(c):
    return 20 * 4 ** c["size"] if c["mesh"] != "torus" else 20 * c["size"] ** 2


def _line_flops(T):
    """A line through a surface of T triangles: at each of two crossings one
    path down an 8-wide tree (8 boxes of 15 operations) and two triangles."""
    return 2 * (math.ceil(math.log(max(T, 8), 8)) * 8 * 15 + 2 * 45) + 600


def work(c):
    path = c["path"]
    net = 2 * (96 * 64 + 3 * 64 * 64 + 64)
    if path == "mlp":
        return dict(bytes=16 * c["points"] + 4 * 18753, flops=c["points"] * (net + 96 * 20 + 256 * 6))
    if path == "train":
        return dict(bytes=16 * c["points"] + 4 * 18753 * 7, flops=3 * c["points"] * net)
    if path == "batch":
        T, Q = c["tri_hi"] / 4.0, c["query_hi"] / 3.0
        return dict(bytes=c["problems"] * (60 * T + 28 * Q),
                    flops=c["problems"] * Q * c["walks"] * 16 * _line_flops(T))
    T = _tris(c)
    Q = c["queries"] or c["grid"] ** 2 * 0.45  # the share of a slice inside the star
    bytes_ = 18 * T + 28 * Q
    if path == "fwd":
        pairs = float(c["paths"]) * c["length"] * Q
        return dict(bytes=bytes_, flops=pairs * 10 + c["paths"] * (c["length"] - 1) * _line_flops(T))
    n = Q * c["walks"] * c["length"]
    if path == "sl":
        return dict(bytes=bytes_, flops=n * max(1, c["ris"]) * 250)
    if path == "nd":
        return dict(bytes=bytes_, flops=n * (_line_flops(T) + 250))
    if path == "cv":
        return dict(bytes=bytes_ + 4 * Q, flops=n * (T * 7 * 12 + _line_flops(T) + net))
    return dict(bytes=bytes_ + (48 * Q if path == "grad" else 0),
                flops=n * _line_flops(T) + (300 * T if path == "setup" else 0))


# ---------------------------------------------------------------- 64 bits
# The library's definitions in plain torch: counter-based streams
# (Philox4x32-10, key (seed ^ problem, seed >> 32), counter (query, walk,
# step << 16 | purpose << 12 | attempt, extra)), lines against every
# triangle, and the walk rules of the entry points.
M32 = 0xFFFFFFFF


def _mul32(a, b):
    lo, hi = (a & 0xFFFF) * b, (a >> 16) * b
    t = hi + (lo >> 16)
    return t >> 16, ((t & 0xFFFF) << 16) | (lo & 0xFFFF)


def _philox(q, w, step, purpose, attempt, extra, seed, problem=0):
    q, w, step, attempt, extra = torch.broadcast_tensors(
        *(torch.as_tensor(t, dtype=torch.int64, device="cuda") for t in (q, w, step, attempt, extra)))
    x, y, z, t = q, w, (step << 16) | (purpose << 12) | attempt, extra
    k0, k1 = (seed & M32) ^ problem, (seed >> 32) & M32
    for _ in range(10):
        h0, l0 = _mul32(0xD2511F53, x)
        h1, l1 = _mul32(0xCD9E8D57, z)
        x, y, z, t = h1 ^ y ^ k0, l1, h0 ^ t ^ k1, l0
        k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
    return x, y, z, t


def _u24(x):
    return (x >> 8).double() * 2.0 ** -24


def _u53(hi, lo):
    return ((hi << 21) | (lo >> 11)).double() * 2.0 ** -53


def _axis(q, w, step, seed, problem=0):
    """Marsaglia's uniform axis, first accepted pair of the stream."""
    n = q.shape[0]
    d = torch.zeros(n, 3, dtype=torch.float64, device="cuda")
    d[:, 2] = 1.0
    left = torch.arange(n, device="cuda")
    for call in range(256):
        if left.numel() == 0:
            break
        u = _philox(q[left], w[left], step, 0, call, 0, seed, problem)
        for a in (0, 2):
            A, B = (2 * (t >> 8) - (1 << 24) + 1 for t in (u[a], u[a + 1]))
            S = A * A + B * B
            if a == 0:
                A0, B0, S0 = A, B, S
        ok0 = S0 < (1 << 48)
        A, B, S = (torch.where(ok0, s, t) for s, t in ((A0, A), (B0, B), (S0, S)))
        ok = S < (1 << 48)
        s = S.double() * 2.0 ** -48
        root = torch.sqrt(1.0 - s) * 2.0
        new = torch.stack([A.double() * 2.0 ** -24 * root, B.double() * 2.0 ** -24 * root, 1 - 2 * s], 1)
        d[left[ok]] = new[ok]
        left = left[~ok]
    return d


class _Surface:
    def __init__(self, v, f):
        v, f = torch.from_numpy(v).cuda().double(), torch.from_numpy(f).cuda().long()
        self.f, self.T = f, f.shape[0]
        self.v0 = v[f[:, 0]]
        self.e1, self.e2 = v[f[:, 1]] - self.v0, v[f[:, 2]] - self.v0
        self.N = torch.linalg.cross(self.e1, self.e2)
        nl = self.N.norm(dim=1)
        self.n, self.area = self.N / nl[:, None], 0.5 * nl
        self.cdf = self.area.cumsum(0)
        self.total = float(self.cdf[-1])
        self.U = torch.cat([-torch.linalg.cross(self.e2, self.v0), self.e2], 1).t().contiguous()
        self.V = torch.cat([-torch.linalg.cross(self.v0, self.e1), -self.e1], 1).t().contiguous()
        self.Nt = -self.N.t().contiguous()

    def lines(self, o, d, own, q, w, step, seed, problem=0):
        """All hits of each line but on triangle `own`, one picked by the
        smallest key: (m, triangle or -1, sign of omega . n, point)."""
        n = o.shape[0]
        od = torch.cat([d, torch.linalg.cross(o, d)], 1)
        ls, ts = [], []
        per = max(1, int(4e7) // self.T)
        for i in range(0, n, per):
            det = d[i:i + per] @ self.Nt
            sg = torch.sign(det)
            a, b = (od[i:i + per] @ self.U) * sg, (od[i:i + per] @ self.V) * sg
            hit = (a >= 0) & (b >= 0) & (a + b <= det.abs()) & (sg != 0)
            l, t = hit.nonzero(as_tuple=True)
            keep = t != own[i + l]
            ls.append(l[keep] + i)
            ts.append(t[keep])
        l, t = torch.cat(ls), torch.cat(ts)
        m = torch.bincount(l, minlength=n)
        k = _philox(q[l], w[l], step, 1, 0, t, seed, problem)
        key = ((k[0] - (1 << 31)) << 32) | k[1]
        best = torch.full((n,), (1 << 63) - 1, dtype=torch.int64, device="cuda")
        best.scatter_reduce_(0, l, key, "amin")
        tri = torch.full((n,), -1, dtype=torch.int64, device="cuda")
        pick = key == best[l]
        tri[l[pick]] = t[pick]
        j = tri.clamp(min=0)
        dn = (self.N[j] * d).sum(1)
        tt = (self.N[j] * (self.v0[j] - o)).sum(1) / dn
        s = torch.where((tt > 0) == (dn > 0), 1.0, -1.0).double()
        return m, tri, s, o + tt[:, None] * d

    def sample(self, u, cdf=None):
        """Area-uniform point of a stream block: triangle, point, barycentrics."""
        cdf = self.cdf if cdf is None else cdf
        j = torch.searchsorted(cdf, _u53(u[0], u[1]) * cdf[-1], right=True).clamp(max=self.T - 1)
        su, u2 = _u24(u[2]).sqrt(), _u24(u[3])
        b1, b2 = su * (1 - u2), su * u2
        return j, self.v0[j] + b1[:, None] * self.e1[j] + b2[:, None] * self.e2[j], (1 - su, b1, b2)


def _f32(t):
    return [float(np.float32(x)) for x in t]


def _field(a, S, j, y, b=None):
    """Boundary field h at y on triangle j and its gradient (None in P1)."""
    if a["data_mode"] == wob.DATA_VERTEX_P1:
        if b is None:
            p = y - S.v0[j]
            nn = (S.N[j] ** 2).sum(1)
            b1 = (torch.linalg.cross(p, S.e2[j]) * S.N[j]).sum(1) / nn
            b2 = (torch.linalg.cross(S.e1[j], p) * S.N[j]).sum(1) / nn
            b = (1 - b1 - b2, b1, b2)
        vd = a["vertex_data"].double()[S.f[j]]
        return b[0] * vd[:, 0] + b[1] * vd[:, 1] + b[2] * vd[:, 2], None
    if a["data_mode"] == wob.DATA_POINT:
        r = y - torch.tensor(_f32(a["x0"]), dtype=torch.float64, device="cuda")
        rl = r.norm(dim=1)
        return 1 / rl, -r / rl[:, None] ** 3
    c = _f32(a["poly"])
    X, Y, Z = y.unbind(1)
    h = (c[0] + c[1] * X + c[2] * Y + c[3] * Z + c[4] * X * X + c[5] * Y * Y + c[6] * Z * Z
         + c[7] * X * Y + c[8] * Y * Z + c[9] * Z * X)
    g = torch.stack([c[1] + 2 * c[4] * X + c[7] * Y + c[9] * Z, c[2] + 2 * c[5] * Y + c[7] * X + c[8] * Z,
                     c[3] + 2 * c[6] * Z + c[8] * Y + c[9] * X], 1)
    return h, g


def _flux(a, S, j, y, b, bc):
    """h (condition 0), dh/dn (1) or dh/dn + alpha h (2); P1 data as given."""
    h, g = _field(a, S, j, y, b)
    if g is None:
        return h
    dn = (S.n[j] * g).sum(1)
    alpha = float(np.float32(a["alpha"]))
    return torch.where(bc == 0, h, torch.where(bc == 1, dn, dn + alpha * h))


def _walk_ids(Q, N, lo, hi):
    i = torch.arange(lo, hi, device="cuda")
    return i // N, i % N


def _reduce(values, Q, N):
    x = values.reshape(*values.shape[:-1], Q, N)
    return x.mean(-1), x.var(-1)


def _dl_exact(S, a, q, N, M, seed, grad=False, problem=0):
    Q, phi = q.shape[0], float(a["side"])
    qi, w = _walk_ids(Q, N, 0, Q * N)
    x0 = torch.from_numpy(q).cuda().double()[qi]
    val = torch.zeros(Q * N, dtype=torch.float64, device="cuda")
    P, gf = torch.ones_like(val), torch.zeros(3, Q * N, dtype=torch.float64, device="cuda")
    live, x, own = torch.arange(Q * N, device="cuda"), x0, torch.full_like(qi, -1)
    for k in range(M):
        if live.numel() == 0:
            break
        d = _axis(qi[live], w[live], k, seed, problem)
        m, j, s, y = S.lines(x, d, own, qi[live], w[live], k, seed, problem)
        on = m > 0
        live, m, j, s, y, x = live[on], m[on], j[on], s[on], y[on], x[on]
        ms = m.double() * s
        P[live] = 0.5 * ms if k == 0 else P[live] * (-phi * ms)
        if k == 0 and grad:
            om = y - x
            r = om.norm(dim=1)
            om = om / r[:, None]
            wn = (om * S.n[j]).sum(1)
            gf[:, live] = (-(S.n[j] - 3 * wn[:, None] * om) / (r * wn)[:, None]).t()
        val[live] += P[live] * (phi if k == M - 1 else 2 * phi) * _field(a, S, j, y)[0]
        x, own = y, j
    return (*_reduce(val, Q, N), *_reduce(gf * val, Q, N)) if grad else _reduce(val, Q, N)


def _sl_values(S, a, q, qi, w, M, seed):
    n, phi, G4 = qi.shape[0], float(a["side"]), 4 * math.pi
    alpha, ris = float(np.float32(a["alpha"])), max(1, a["ris"])
    mixed = a["kind"] == wob.MIXED_SL
    if mixed:
        k_mix, p_k = _f32((a["k_mix"], a["p_k"]))
        bc_of = a["bc_type"].long()
    x, bx = q[qi], torch.full_like(qi, -1)
    nx, jx = torch.zeros_like(x), torch.zeros_like(qi)
    acc = torch.zeros(n, dtype=torch.float64, device="cuda")
    P, W0, alive = torch.ones_like(acc), torch.zeros_like(acc), torch.ones(n, dtype=torch.bool, device="cuda")

    def kernel(y):
        r = y - x
        rl = r.norm(dim=1)
        G = 1 / (G4 * rl)
        dg = (r * nx).sum(1) / (G4 * rl ** 3)
        K = torch.where(bx < 0, G, torch.where(bx == 1, -2 * phi * dg, -2 * phi * (dg + alpha * G)))
        return torch.where(bx == 0, -(k_mix / p_k) * G, K) if mixed else K

    for k in range(M):
        if ris == 1:
            j, y, b = S.sample(_philox(qi, w, k, 2, 0, 0, seed))
            wf = kernel(y) * S.total
        else:
            ks = torch.stack([kernel(S.sample(_philox(qi, w, k, 2, c, 0, seed))[1]) for c in range(ris)])
            cum = ks.abs().cumsum(0)
            u = _philox(qi, w, k, 5, 0, 0, seed)
            pick = (cum <= _u53(u[0], u[1]) * cum[-1]).sum(0).clamp(max=ris - 1)
            j, y, b = S.sample(_philox(qi, w, k, 2, pick, 0, seed))
            wf = ks.gather(0, pick[None])[0].sign() * S.total * cum[-1] / ris
            alive &= cum[-1] > 0
        if mixed:
            stay = (bx == 0) & (_u24(_philox(qi, w, k, 4, 0, 0, seed)[0]) >= p_k)
            j, y = torch.where(stay, jx, j), torch.where(stay[:, None], x, y)
            wf = torch.where(stay, torch.full_like(wf, 1 / (1 - p_k)), wf)
            by = bc_of[j]
        else:
            by = torch.full_like(j, 2 if a["kind"] == wob.ROBIN_SL else 1)
        if k == 0:
            W0 = wf
        else:
            P = P * wf
        src = _flux(a, S, j, y, b, by) * (torch.where(by == 0, k_mix, 2 * phi) if mixed else 2 * phi)
        acc += torch.where(alive, P * src * (0.5 if k == M - 1 else 1.0), torch.zeros_like(acc))
        x, nx, bx, jx = y, S.n[j], by, j
    return W0 * acc


def _sl_exact(S, a, q, N, M, seed):
    Q, qd = q.shape[0], torch.from_numpy(q).cuda().double()
    step = 1 << 20
    vals = [_sl_values(S, a, qd, *_walk_ids(Q, N, i, min(i + step, Q * N)), M, seed)
            for i in range(0, Q * N, step)]
    return _reduce(torch.cat(vals), Q, N)


def _nd_exact(S, a, q, prim, N, M, seed):
    Q, phi = q.shape[0], float(a["side"])
    qi, w = _walk_ids(Q, N, 0, Q * N)
    x = torch.from_numpy(q).cuda().double()[qi]
    own = torch.from_numpy(prim).cuda().long()[qi]
    on0 = own >= 0
    val = torch.zeros(Q * N, dtype=torch.float64, device="cuda")
    P, alive = torch.ones_like(val), torch.ones_like(on0)
    for k in range(M + 1):
        go = alive if k else alive & ~on0
        i = go.nonzero()[:, 0]
        if i.numel() == 0:
            continue
        j, y, b = S.sample(_philox(qi[i], w[i], k, 2, 0, 0, seed))
        c = (phi if k == 0 else 2 * phi) * (0.5 if k == M else 1.0)
        f = _flux(a, S, j, y, b, torch.ones_like(j))
        val[i] += P[i] * c * S.total * f / (4 * math.pi * (y - x[i]).norm(dim=1))
        if k == M:
            break
        d = _axis(qi[i], w[i], k, seed)
        m, t, s, y = S.lines(x[i], d, own[i], qi[i], w[i], k, seed)
        P[i] *= (0.5 if k == 0 else 1.0) * phi * m.double() * s
        alive[i[m == 0]] = False
        x[i], own[i] = y, t
    return _reduce(val, Q, N)


def _fwd_exact(S, a, q, n, M, seed):
    phi, beta = float(a["side"]), float(np.float32(0.1))
    third = torch.full((S.T,), 1.0 / 3.0, dtype=torch.float64, device="cuda")
    qc = _field(a, S, torch.arange(S.T, device="cuda"), None, (third, third, third))[0].abs() * S.area
    cdf = (qc + beta * (qc.sum() / S.total) * S.area).cumsum(0)
    p = torch.arange(n, device="cuda")
    w = torch.full_like(p, M32)
    j, z, b = S.sample(_philox(p, w, 0, 2, 0, 0, seed), cdf)
    wt = torch.diff(cdf, prepend=cdf.new_zeros(1))[j]
    amp = 2 * phi * _field(a, S, j, z, b)[0] * S.area[j] * cdf[-1] / wt
    pos, wts = torch.zeros(M, n, 3, dtype=torch.float64, device="cuda"), torch.zeros(M, n, dtype=torch.float64, device="cuda")
    for k in range(M):
        pos[k], wts[k] = z, amp * (0.5 if k == M - 1 else 1.0)
        if k == M - 1:
            break
        m, t, s, y = S.lines(z, _axis(p, w, k, seed), j, p, w, k, seed)
        amp = amp * phi * m.double() * s
        hit = m > 0
        z, j = torch.where(hit[:, None], y, z), torch.where(hit, t, j)
    qd = torch.from_numpy(q).cuda().double()
    est, var = torch.empty(2, qd.shape[0], dtype=torch.float64, device="cuda")
    per = max(1, int(2e8) // (M * n))
    flat = pos.reshape(-1, 3)
    for i in range(0, qd.shape[0], per):
        r2 = sum((qd[i:i + per, None, c] - flat[None, :, c]) ** 2 for c in range(3))
        v = (r2.rsqrt_().reshape(-1, M, n) * (wts / (4 * math.pi))).sum(1)
        est[i:i + per], var[i:i + per] = v.mean(1), v.var(1)
    return dict(est=est, var=var)


def _network(params):
    """Forward of the 96 -> 4 x 64 -> 1 network; returns (layers, call)."""
    p, o, layers = params.double(), 0, []
    for i, k in ((96, 64), (64, 64), (64, 64), (64, 64), (64, 1)):
        layers.append((p[o:o + i * k].reshape(k, i), p[o + i * k:o + i * k + k]))
        o += i * k + k

    def call(x):
        f = 2.0 ** (torch.arange(16, device="cuda", dtype=torch.float64) / 3)
        t = 2 * math.pi * x.double()[:, :, None] * f
        h = torch.stack([t.sin(), t.cos()], -1).reshape(len(x), 96)
        for n, (W, b) in enumerate(layers):
            h = h @ W.t() + b
            if n < 4:
                h = h * torch.sigmoid(h)
        return h[:, 0]

    return layers, call


def _train_exact(c, seed):
    p, m, v, x, t = (y.double() for y in _train_state(c, seed))
    with torch.enable_grad():
        w = p.clone().requires_grad_()
        loss = ((_network(w)[1](x) - t) ** 2).mean()
        grad, = torch.autograd.grad(loss, w)
    b1, b2, eps, lr = _f32((0.9, 0.999, 1e-8, 1e-3))
    m, v = b1 * m + (1 - b1) * grad, b2 * v + (1 - b2) * grad * grad
    p = p - lr * (m / (1 - b1 ** 1000)) / ((v / (1 - b2 ** 1000)).sqrt() + eps)
    return p, m, v, grad, loss.detach()[None]


def _rule(level):
    """Radon's seven nodes (barycentrics, weights), on 4^level parts."""
    s = math.sqrt(15.0)
    a1, b1, a2, b2 = (6 - s) / 21, (9 + 2 * s) / 21, (6 + s) / 21, (9 - 2 * s) / 21
    P = np.array([[1 / 3] * 3, [b1, a1, a1], [a1, b1, a1], [a1, a1, b1], [b2, a2, a2], [a2, b2, a2], [a2, a2, b2]])
    W = np.array([9 / 40] + [(155 - s) / 1200] * 3 + [(155 + s) / 1200] * 3)
    parts = [np.eye(3)]
    for _ in range(level):
        cut = []
        for A, B, C in parts:
            ab, bc, ca = (A + B) / 2, (B + C) / 2, (C + A) / 2
            cut += [np.stack(t) for t in ((A, ab, ca), (B, bc, ab), (C, ca, bc), (ab, bc, ca))]
        parts = cut
    B = np.concatenate([P @ t for t in parts])
    return (torch.from_numpy(B).cuda(), torch.from_numpy(np.tile(W, len(parts)) / len(parts)).cuda())


def _quad(S, net, x, own, fx):
    """-int dG/dn_y (f - fx) dA by the rule, level 2 near the target."""
    cen = S.v0 + (S.e1 + S.e2) / 3
    edge = torch.stack([S.e1.norm(dim=1), S.e2.norm(dim=1), (S.e2 - S.e1).norm(dim=1)]).amax(0)
    rules = []
    for level in (0, 2):
        B, W = _rule(level)
        y = S.v0[:, None] + B[None, :, 1, None] * S.e1[:, None] + B[None, :, 2, None] * S.e2[:, None]
        rules.append((y, W, net(y.reshape(-1, 3)).reshape(S.T, -1)))
    out = torch.zeros(len(x), dtype=torch.float64, device="cuda")
    skip = torch.full((len(x),), -1, device="cuda") if own is None else own
    per = max(1, int(4e6) // S.T)
    for i in range(0, len(x), per):
        p, o = x[i:i + per], skip[i:i + per]
        f0 = torch.zeros(len(p), dtype=torch.float64, device="cuda") if fx is None else fx[i:i + per]
        near = torch.cdist(p, cen, compute_mode="donot_use_mm_for_euclid_dist") < 2 * edge
        dot = ((S.v0 * S.n).sum(1) - p @ S.n.t()) * S.area
        y, W, f = rules[0]
        s = torch.zeros_like(dot)
        for c in range(7):
            ri = sum((y[None, :, c, d] - p[:, None, d]) ** 2 for d in range(3)).rsqrt_()
            s += W[c] * (f[None, :, c] - f0[:, None]) * ri ** 3
        l, t = near.nonzero(as_tuple=True)
        y, W, f = rules[1]
        for a in range(0, len(l), 100000):
            la, ta = l[a:a + 100000], t[a:a + 100000]
            ri = (y[ta] - p[la][:, None]).norm(dim=2).reciprocal()
            s[la, ta] = (W * (f[ta] - f0[la][:, None]) * ri ** 3).sum(1)
        s *= dot
        at = (o >= 0).nonzero()[:, 0]
        s[at, o[at]] = 0
        out[i:i + per] = s.sum(1) / (4 * math.pi)
    return out


def _cv_exact(S, a, q, N, M, seed):
    net = _network(wob.mlp_init(seed))[1]
    Q = q.shape[0]
    qd = torch.from_numpy(q).cuda().double()
    qi, w = _walk_ids(Q, N, 0, Q * N)
    val = torch.zeros(Q * N, dtype=torch.float64, device="cuda")
    P, live, x, own = torch.ones_like(val), torch.arange(Q * N, device="cuda"), qd[qi], torch.full_like(qi, -1)
    for k in range(M):
        m, j, s, y = S.lines(x, _axis(qi[live], w[live], k, seed), own, qi[live], w[live], k, seed)
        on = m > 0
        live, m, j, s, y = live[on], m[on], j[on], s[on], y[on]
        ms = m.double() * s
        P[live] = 0.5 * ms if k == 0 else P[live] * -ms
        nu = net(y)
        h = -2 * _quad(S, net, y, j, nu) - nu
        r = 2 * _field(a, S, j, y)[0] - nu + h
        val[live] += P[live] * (0.5 if k == M - 1 else 1.0) * r
        x, own = y, j
    val = val.reshape(Q, N)
    return torch.stack([val.sum(1), (val ** 2).sum(1)]), _quad(S, net, qd, None, None)


def exact(c, seed):
    path = c["path"]
    if path == "mlp":
        x, _ = _sphere_points(c["points"], seed)
        net = _network(wob.mlp_init(seed))[1]
        return torch.cat([net(t) for t in x.split(1 << 17)])
    if path == "train":
        return _train_exact(c, seed)
    if path == "batch":
        items = _batch_items(c, seed)
        if sum(float(len(it.tris)) * len(it.queries) * c["walks"] * it.max_len for it in items) > MAX_PAIRS:
            return None
        a = dict(side=1, data_mode=wob.DATA_POINT, x0=X_SIDE)
        out = [_dl_exact(_Surface(it.verts, it.tris), a, it.queries, c["walks"], it.max_len, seed, problem=i)
               for i, it in enumerate(items)]
        return torch.cat([e for e, _ in out]), torch.cat([v for _, v in out])
    n = c.get("walks", 1) * (c["queries"] or c.get("grid", 0) ** 2)
    lines = float(n * c["length"] if path != "fwd" else c["paths"] * (c["length"] - 1))
    if path != "sl" and lines * _tris(c) > MAX_PAIRS:
        return None  # too many pairs for brute force
    if path == "cv" and lines * _tris(c) * 7 > MAX_PAIRS:
        return None
    v, f, a, q, prim = _scene(c, seed)
    S = _Surface(v, f)
    if path == "sl":
        return _sl_exact(S, a, q, c["walks"], c["length"], seed)
    if path == "nd":
        return _nd_exact(S, a, q, prim, c["walks"], c["length"], seed)
    if path == "fwd":
        return _fwd_exact(S, a, q, c["paths"], c["length"], seed)
    if path == "cv":
        return _cv_exact(S, a, q, c["walks"], c["length"], seed)
    r = _dl_exact(S, a, q, c["walks"], c["length"], seed, grad=path == "grad")
    return r if path != "grad" else dict(est=r[0], var=r[1], grad_est=r[2], grad_var=r[3])
