"""Performance cases: the evaluations a user of the library asks for.

Every case goes through the package's public entry points with a plan, batch
or potential that a program keeps between calls, and device buffers it owns.
The meshes are the paper's bodies (cube, sphere, thin plate, torus, and the
tetrahedral ball of the scalar potential), in the sizes of the repository's
benchmark, serving pool and tests; the fields are seeded smooth unit
magnetisations (or the charges such a field has), different for every seed.

A case is a dict:
  form      eval (slp_eval), states (slp_eval_states), probe
            (slp_eval_probe), batched (slp_eval_batched), potential
            (slp_potential_eval)
  mesh      cube, sphere, plate, torus; ball for the potential
  size      squares per cube edge; icosphere level; plate cells along its
            length; torus segments along its tube; ball core cells (even)
  rule      quadrature points per triangle (1, 3, 7)
  input     nodal, sigma, mag, element
  bits, tol precision and tolerance of the plan
  grid      "" (automatic) or "LxxLyxLz"
  options   "" , "triangles" (triangle integrals) or "deterministic"
  count     states of a states call, states per mesh of a batched call,
            probe points of a probe call; else 1
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1305_3162_gb300 as slp

DEVICE = "cuda"
INPUT = {"nodal": slp.SLP_INPUT_NODAL_MAG, "sigma": slp.SLP_INPUT_SIGMA, "mag": slp.SLP_INPUT_MAG,
         "element": slp.SLP_INPUT_ELEMENT}
#: pairs (target, source) up to which the 64-bit direct sum stays well under its time
PAIRS = 1.2e11
TRIANGLE_PAIRS = 2.5e9


def _case(name, form, mesh, size, rule=3, input="nodal", bits=32, tol=1e-5, grid="", options="", count=1):
    c = {"form": form, "mesh": mesh, "size": size, "rule": rule, "input": input, "bits": bits, "tol": tol,
         "grid": grid, "options": options, "count": count}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a coarse cube in a double-precision study (latency)
        _case("cube8 fp64", "eval", "cube", 8, bits=64, tol=1e-10, grid="32x32x32"),
        # a small sphere inside an outer loop: launches and latency count
        _case("sphere3", "eval", "sphere", 3, rule=7),
        # the benchmark's evaluation: one state of the level-5 sphere
        _case("sphere5", "eval", "sphere", 5, rule=7, grid="128x128x128"),
        # charges at the quadrature points (g of a coupled solver): near field per pair
        _case("sphere5 sigma", "eval", "sphere", 5, rule=7, input="sigma", grid="128x128x128"),
        # element-wise charges with exact triangle integrals, the paper's own discretisation
        _case("sphere5 triangles", "eval", "sphere", 5, rule=7, input="element", grid="128x128x128",
              options="triangles"),
        # double precision at a size that needs the radial kernel
        _case("sphere4 fp64", "eval", "sphere", 4, rule=7, bits=64, tol=1e-10, grid="128x128x128"),
        # eight states of one mesh in one call (field sweep, serving)
        _case("torus400 states", "states", "torus", 400, count=8, grid="256x256x128"),
        # uneven meshes, several states each, in one batched call
        _case("mixed batched", "batched", "cube", 32, count=4),
        # a thin film: near field dominates
        _case("plate400", "eval", "plate", 400, grid="512x128x16"),
        # the largest call: a finely meshed cube
        _case("cube200", "eval", "cube", 200, grid="512x512x512"),
        # the whole scalar potential of a tetrahedral ball, small and large
        _case("ball16 potential", "potential", "ball", 16, input="nodal"),
        _case("ball32 potential", "potential", "ball", 32, input="nodal"),
    ]


def _spread(rng, lo, hi):
    """An integer between lo and hi, uniform over its logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    form = rng.choice(["eval", "eval", "eval", "eval", "states", "batched", "probe", "potential"])
    bits = rng.choice([32, 32, 32, 64])
    tol = 1e-5 if bits == 32 else 1e-10
    if form == "potential":
        return _case("", form, "ball", 2 * _spread(rng, 3, 16 if bits == 32 else 6), bits=bits, tol=tol)
    if form == "batched":
        return _case("", form, "cube", _spread(rng, 7, 32), count=rng.randint(1, 4))
    mesh = rng.choice(["cube", "sphere", "plate", "torus"])
    low = {"cube": 6, "sphere": 2, "plate": 20, "torus": 30}
    if bits == 64:  # double-precision studies are on coarse meshes
        top = {"cube": 14, "sphere": 3, "plate": 25, "torus": 40}
    elif form == "states":
        top = {"cube": 26, "sphere": 4, "plate": 90, "torus": 130}
    else:
        top = {"cube": 150, "sphere": 6, "plate": 300, "torus": 400}
    size = rng.randint(low[mesh], top[mesh]) if mesh == "sphere" else _spread(rng, low[mesh], top[mesh])
    small = size <= {"cube": 50, "sphere": 5, "plate": 150, "torus": 200}[mesh]
    rule = rng.choice([1, 3, 3, 7]) if small else rng.choice([1, 3, 3])
    grid = rng.choice(["", "128x128x128"]) if small else ""
    if form == "states":
        return _case("", form, mesh, size, rule=rule, bits=bits, tol=tol, grid=grid, count=rng.randint(2, 20))
    if form == "probe":
        return _case("", form, mesh, size, rule=rule, bits=bits, tol=tol, grid=grid, count=_spread(rng, 500, 20000))
    options = rng.choice(["", "", "", "deterministic", "triangles"]) if small else ""
    if options == "triangles":  # wants triangles of at most 24 - 2m grid cells
        size, grid = max(size, 3), "128x128x128"
    kind = rng.choice(["nodal", "element"] if options == "triangles" else ["nodal", "nodal", "sigma", "mag"])
    return _case("", form, mesh, size, rule=rule, input=kind, bits=bits, tol=tol, grid=grid, options=options)


# ------------------------------------------------------------------ meshes
def _box(lx, ly, lz, nx, ny, nz):
    """Surface of a centred cuboid, nx x ny x nz squares per edge, two triangles per square."""
    n = np.array([nx, ny, nz])
    I = np.stack(np.meshgrid(*[np.arange(k + 1) for k in n], indexing="ij"), -1).reshape(-1, 3)
    on = ((I == 0) | (I == n)).any(1)
    number = np.cumsum(on) - 1
    V = I[on] / n * np.array([lx, ly, lz]) - 0.5 * np.array([lx, ly, lz])
    stride = np.array([(ny + 1) * (nz + 1), nz + 1, 1])
    T = []
    for axis in range(3):
        for high in (0, 1):
            a, b = (axis + 1) % 3, (axis + 2) % 3
            if not high:
                a, b = b, a
            i, j = (x.ravel() for x in np.meshgrid(np.arange(n[a]), np.arange(n[b]), indexing="ij"))
            p = high * n[axis] * stride[axis] + i * stride[a] + j * stride[b]
            q = [number[p], number[p + stride[a]], number[p + stride[a] + stride[b]], number[p + stride[b]]]
            T += [np.stack([q[0], q[1], q[2]], 1), np.stack([q[0], q[2], q[3]], 1)]
    return V, np.concatenate(T).astype(np.int32)


def _sphere(level):
    """Icosahedron bisected `level` times onto the unit sphere."""
    t = (1 + 5 ** 0.5) / 2
    V = np.array([[-1, t, 0], [1, t, 0], [-1, -t, 0], [1, -t, 0], [0, -1, t], [0, 1, t], [0, -1, -t], [0, 1, -t],
                  [t, 0, -1], [t, 0, 1], [-t, 0, -1], [-t, 0, 1]])
    V /= np.linalg.norm(V, axis=1, keepdims=True)
    F = np.array([[0, 11, 5], [0, 5, 1], [0, 1, 7], [0, 7, 10], [0, 10, 11], [1, 5, 9], [5, 11, 4], [11, 10, 2],
                  [10, 7, 6], [7, 1, 8], [3, 9, 4], [3, 4, 2], [3, 2, 6], [3, 6, 8], [3, 8, 9], [4, 9, 5], [2, 4, 11],
                  [6, 2, 10], [8, 6, 7], [9, 8, 1]])
    for _ in range(level):
        n, m = len(V), len(F)
        e = np.sort(np.concatenate([F[:, [0, 1]], F[:, [1, 2]], F[:, [2, 0]]]), 1)
        key, at = np.unique(e[:, 0] * n + e[:, 1], return_inverse=True)
        mid = V[key // n] + V[key % n]
        V = np.concatenate([V, mid / np.linalg.norm(mid, axis=1, keepdims=True)])
        ab, bc, ca = (n + at.ravel()[k * m:(k + 1) * m] for k in range(3))
        F = np.concatenate([np.stack(f, 1) for f in ((F[:, 0], ab, ca), (F[:, 1], bc, ab), (F[:, 2], ca, bc),
                                                     (ab, bc, ca))])
    return V, F.astype(np.int32)


def _torus(nu, nv):
    """Torus of radii 2 and 0.5, nu x nv quadrilaterals."""
    u, v = np.meshgrid(2 * np.pi * np.arange(nu) / nu, 2 * np.pi * np.arange(nv) / nv, indexing="ij")
    r = 2 + 0.5 * np.cos(v)
    V = np.stack([r * np.cos(u), r * np.sin(u), 0.5 * np.sin(v)], -1).reshape(-1, 3)
    i, j = (x.ravel() for x in np.meshgrid(np.arange(nu), np.arange(nv), indexing="ij"))
    p, q = i * nv, (i + 1) % nu * nv
    k = (j + 1) % nv
    return V, np.concatenate([np.stack([p + j, q + j, q + k], 1), np.stack([p + j, q + k, p + k], 1)]).astype(np.int32)


def _surface(mesh, size):
    if mesh == "cube":
        return _box(1, 1, 1, size, size, size)
    if mesh == "sphere":
        return _sphere(size)
    if mesh == "plate":  # 2000 x 500 x 20, square cells
        return _box(2000, 500, 20, size, max(1, size // 4), max(1, size // 100))
    return _torus(size, max(8, size // 4))


def _ball(n, radius=0.2):
    """Tetrahedra of a ball: a core cube of n^3 cells and n / 2 layers of n x n
    cells over each of its faces out to the sphere, each cell cut into the six
    tetrahedra along its diagonal (index coordinates along the global axes and
    outward, so neighbours cut shared faces alike)."""
    h, layers = n // 2, n // 2
    w = n + 1

    def key(q, k):
        return (((q[..., 0] + h) * w + q[..., 1] + h) * w + q[..., 2] + h) * (layers + 1) + k

    paths = []
    for order in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
        corner, path = [0, 0, 0], [(0, 0, 0)]
        for axis in order:
            corner[axis] = 1
            path.append(tuple(corner))
        paths.append(path)
    tets = []
    core = np.stack(np.meshgrid(*[np.arange(-h, h)] * 3, indexing="ij"), -1).reshape(-1, 3)
    tets += [np.stack([key(core + c, 0) for c in path], 1) for path in paths]
    for axis in range(3):
        a, b = [d for d in range(3) if d != axis]
        for side in (-h, h):
            u, v, k = (x.ravel() for x in np.meshgrid(np.arange(-h, h), np.arange(-h, h), np.arange(layers),
                                                      indexing="ij"))
            q = np.zeros((u.size, 3), dtype=np.int64)
            for path in paths:
                cols = []
                for du, dv, dk in path:
                    q[:, axis], q[:, a], q[:, b] = side, u + du, v + dv
                    cols.append(key(q, k + dk))
                tets.append(np.stack(cols, 1))
    keys, at = np.unique(np.concatenate(tets), return_inverse=True)
    tets = at.reshape(-1, 4)
    k = keys % (layers + 1)
    q = keys // (layers + 1)
    q = np.stack([q // (w * w), q // w % w, q % w], 1) - h
    p = q * (0.5 * radius / h)
    t = (k / layers)[:, None]
    X = (1 - t) * p + t * radius * p / np.maximum(np.linalg.norm(p, axis=1, keepdims=True), 1e-300)
    e = X[tets[:, 1:]] - X[tets[:, :1]]
    flip = np.einsum("ij,ij->i", e[:, 0], np.cross(e[:, 1], e[:, 2])) < 0
    tets[flip, 2], tets[flip, 3] = tets[flip, 3].copy(), tets[flip, 2].copy()
    return X, tets.astype(np.int32)


def _parts(case):
    """(V, T, rule) of a batched call's meshes: a cube, a sphere, a torus and a plate of uneven sizes."""
    n = case["size"]
    level = max(2, min(5, int(round(math.log(0.6 * n * n, 4)))))
    return [(*_surface("cube", n), 3), (*_sphere(level), 7), (*_torus(2 * n, max(8, n // 2)), 3),
            (*_surface("plate", 4 * n), 3)]


# ------------------------------------------------------------------ inputs
def _field(V, seed):
    """Smooth unit magnetisation at the points V: eight seeded cosine modes of
    the bounding box and a little noise (float64, on the GPU)."""
    rng = np.random.default_rng(seed)
    x = torch.as_tensor(V, dtype=torch.float64, device=DEVICE)
    lo = x.min(0).values
    x = (x - lo) / (x.max(0).values - lo).clamp_min(1e-30)
    m = torch.zeros_like(x)
    for _ in range(8):
        k, a, p = rng.integers(-2, 3, size=3), rng.normal(size=3), rng.uniform(0, 2 * np.pi)
        c = torch.cos(2 * math.pi * (x @ torch.as_tensor(k, dtype=torch.float64, device=DEVICE)) + p)
        m += torch.as_tensor(a, device=DEVICE) * c[:, None]
    g = torch.Generator(device=DEVICE).manual_seed(int(rng.integers(1 << 40)))
    m += 1e-3 * torch.randn(x.shape, generator=g, device=DEVICE, dtype=torch.float64)
    return m / m.norm(dim=1, keepdim=True)


def _rule(q):
    """Barycentric points and weights of the library's rules, in its order (slp.h)."""
    if q == 1:
        return np.full((1, 3), 1 / 3), np.ones(1)
    if q == 3:
        return np.array([[2 / 3, 1 / 6, 1 / 6], [1 / 6, 2 / 3, 1 / 6], [1 / 6, 1 / 6, 2 / 3]]), np.full(3, 1 / 3)
    s = math.sqrt(15.0)
    lam, w = [[1 / 3] * 3], [9 / 40]
    for a, wa in (((6 - s) / 21, (155 - s) / 1200), ((6 + s) / 21, (155 + s) / 1200)):
        lam += [[a, a, 1 - 2 * a], [a, 1 - 2 * a, a], [1 - 2 * a, a, a]]
        w += [wa] * 3
    return np.array(lam), np.array(w)


def _points(V, T, q):
    """Quadrature points, their weights w |S|, and the triangles' outward normals (float64, on the GPU)."""
    lam, w = (torch.as_tensor(x, device=DEVICE) for x in _rule(q))
    P = torch.as_tensor(V, device=DEVICE)[torch.as_tensor(T, device=DEVICE).long()]
    n = torch.linalg.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
    area2 = n.norm(dim=1, keepdim=True)
    y = torch.einsum("sa,tad->tsd", lam, P).reshape(-1, 3)
    return y, (0.5 * area2 * w).reshape(-1), n / area2


def _input(case, V, T, seed):
    """One state's input in the plan's precision."""
    dt = torch.float64 if case["bits"] == 64 else torch.float32
    kind = case["input"]
    if kind == "nodal":
        x = _field(V, seed)
    elif kind == "element":
        y, _, n = _points(V, T, 1)
        x = (_field(y, seed) * n).sum(1)
    else:
        y, _, n = _points(V, T, case["rule"])
        x = _field(y, seed)
        if kind == "sigma":
            x = (x * n.repeat_interleave(case["rule"], 0)).sum(1)
    return x.to(dt).contiguous()


def _inside(mesh, V, T, count):
    """Points inside the body: seeded surface points drawn towards its centre
    (a torus: towards the circle of its tube)."""
    rng = np.random.default_rng(17)
    t = T[rng.integers(0, len(T), count)]
    p = np.einsum("ka,kad->kd", rng.dirichlet(np.ones(3), count), V[t])
    core = np.zeros((count, 3))
    if mesh == "torus":
        core[:, :2] = 2 * p[:, :2] / np.hypot(p[:, 0], p[:, 1])[:, None]
    return core + rng.uniform(0.05, 0.95, (count, 1)) * (p - core)


# ------------------------------------------------------------------ states
class _Probe:
    """A plan with a probe set, released in order."""

    def __init__(self, plan, points):
        self.plan = plan
        self.handle = slp.slp_probe_create(plan.handle, points)

    def __del__(self):
        slp.slp_probe_destroy(self.handle)
        self.plan.close()


class _Potential:
    def __init__(self, X, K, tol, opts):
        self.handle = slp.slp_potential_create(X, K, tol, opts)

    def __del__(self):
        slp.slp_potential_destroy(self.handle)


def _grid(case):
    return tuple(int(x) for x in case["grid"].split("x")) if case["grid"] else None


def _plan(case, V, T, rule):
    return slp.Plan(V, T, quadrature=rule, tolerance=case["tol"], precision=case["bits"], grid=_grid(case),
                    deterministic=case["options"] == "deterministic", integration=int(case["options"] == "triangles"))


def prepare(case, seed):
    dt = torch.float64 if case["bits"] == 64 else torch.float32
    st = {"form": case["form"], "kind": INPUT[case["input"]], "count": case["count"]}
    if case["form"] == "potential":
        X, K = _ball(case["size"])
        o = slp.slp_default_opts()
        o.precision = case["bits"]
        st["pot"] = _Potential(X, K, case["tol"], o)
        st["in"] = _field(X, seed).to(dt).contiguous()
        st["phi"] = torch.empty(len(X), dtype=dt, device=DEVICE)
        st["phi1"] = torch.empty(len(X), dtype=dt, device=DEVICE)
        return st
    if case["form"] == "batched":
        parts = _parts(case)
        st["plans"] = [_plan(case, V, T, q) for V, T, q in parts]
        st["in"] = [torch.stack([_input(case, V, T, (seed, i, k)) for k in range(case["count"])])
                    for i, (V, T, q) in enumerate(parts)]
        st["phi"] = [torch.empty(case["count"], len(V), dtype=dt, device=DEVICE) for V, T, q in parts]
        return st
    V, T = _surface(case["mesh"], case["size"])
    st["plan"] = _plan(case, V, T, case["rule"])
    if case["form"] == "states":
        st["in"] = torch.stack([_input(case, V, T, (seed, k)) for k in range(case["count"])])
        st["phi"] = torch.empty(case["count"], len(V), dtype=dt, device=DEVICE)
        return st
    st["in"] = _input(case, V, T, seed)
    st["phi"] = torch.empty(len(V), dtype=dt, device=DEVICE)
    if case["form"] == "probe":
        st["probe"] = _Probe(st["plan"], _inside(case["mesh"], V, T, case["count"]))
        st["phi_points"] = torch.empty(case["count"], dtype=dt, device=DEVICE)
    return st


def run(st):
    stream = torch.cuda.current_stream()
    form = st["form"]
    if form == "eval":
        st["plan"].eval(st["kind"], st["in"], st["phi"], stream)
        return st["phi"]
    if form == "states":
        slp.slp_eval_states(st["plan"].handle, st["kind"], st["count"], st["in"], st["phi"], stream)
        return st["phi"]
    if form == "probe":
        slp.slp_eval_probe(st["plan"].handle, st["probe"].handle, st["kind"], st["in"], st["phi"], st["phi_points"],
                           stream)
        return [st["phi"], st["phi_points"]]
    if form == "batched":
        slp.slp_eval_batched([p.handle for p in st["plans"]], st["kind"], st["in"], st["phi"],
                             [st["count"]] * len(st["plans"]), stream)
        return st["phi"]
    slp.slp_potential_eval(st["pot"].handle, st["in"], st["phi"], st["phi1"], stream)
    return [st["phi"], st["phi1"]]


# ------------------------------------------------------------------ work
def work(case):
    """Coordinates and charge of every source and coordinates and potential of
    every target once, the input once; the window products of spread and
    interpolation (2m points per axis).  The potential: the mesh, m and phi."""
    es = case["bits"] // 8
    if case["form"] == "potential":
        X, K = _ball(case["size"])
        return {"bytes": len(X) * (24 + 5 * es) + 16 * len(K), "flops": 30.0 * len(K)}
    box = (2 * (4 if case["bits"] == 32 else 7)) ** 3
    total = {"bytes": 0.0, "flops": 0.0}
    parts = _parts(case) if case["form"] == "batched" else [(*_surface(case["mesh"], case["size"]), case["rule"])]
    states = case["count"] if case["form"] in ("states", "batched") else 1
    for V, T, q in parts:
        n, s = len(V), len(T) * q
        if case["form"] == "probe":
            n += case["count"]
        values = {"nodal": 3 * len(V), "sigma": s, "mag": 3 * s, "element": len(T)}[case["input"]]
        total["bytes"] += es * (3 * (s + n) + states * (values + n))
        total["flops"] += states * 2.0 * box * (s + n)
    return total


# ------------------------------------------------------------------ 64-bit values
def _direct(x, y, qk):
    """(1 / 4 pi) sum_k qk / |x - y_k| for every x, in 64 bits; qk [Q] or [Q][states]."""
    qk = qk.reshape(len(y), -1)
    out = torch.empty(len(x), qk.shape[1], dtype=torch.float64, device=DEVICE)
    yt = y.t().contiguous()
    rows = max(1, (1 << 24) // len(y))
    a, b = (torch.empty(rows, len(y), dtype=torch.float64, device=DEVICE) for _ in range(2))
    for i in range(0, len(x), rows):
        p = x[i:i + rows]
        d, t = a[:len(p)], b[:len(p)]
        torch.sub(p[:, :1], yt[0], out=d)
        d.mul_(d)
        for c in (1, 2):
            torch.sub(p[:, c:c + 1], yt[c], out=t)
            d.addcmul_(t, t)
        torch.mm(d.rsqrt_(), qk, out=out[i:i + rows])
    return (out / (4 * math.pi)).squeeze(1)


def _triangles(x, P, n, g):
    """(1 / 4 pi) sum_j g_j int_{S_j} 1 / |x - y| dA for every x, each integral
    in closed form: the sum over a triangle's edges of the logarithm and the
    solid-angle terms of the uniform potential of a polygon."""
    out = torch.empty(len(x), dtype=torch.float64, device=DEVICE)
    rows = max(1, (1 << 23) // len(P))
    edges = []
    for k in range(3):
        a, b = P[:, k], P[:, (k + 1) % 3]
        length = (b - a).norm(dim=1, keepdim=True)
        e = (b - a) / length
        u = torch.linalg.cross(e, n)  # in the plane, outward of the edge
        edges.append((e, (a * e).sum(1), (b * e).sum(1), u, (a * u).sum(1), 1e-13 * length.ravel()))
    off = (P[:, 0] * n).sum(1)
    for i in range(0, len(x), rows):
        p = x[i:i + rows]
        d = (p @ n.t() - off).abs()
        total = torch.zeros_like(d)
        for e, a, b, u, c, tiny in edges:
            s = p @ e.t()
            lo, hi = a - s, b - s
            t = c - p @ u.t()
            r02 = t * t + d * d
            rl, rh = (lo * lo + r02).sqrt_(), (hi * hi + r02).sqrt_()
            num = torch.where(hi >= 0, rh + hi, r02 / (rh - hi))
            den = torch.where(lo >= 0, rl + lo, r02 / (rl - lo))
            term = t * torch.log(num / den) - d * (torch.atan2(t * hi, r02 + d * rh) - torch.atan2(t * lo, r02 + d * rl))
            total += torch.where(t.abs() > tiny, term, torch.zeros_like(term))
        torch.mv(total, g, out=out[i:i + rows])
    return out / (4 * math.pi)


def _exact_points(case, V, T, rule, x, inputs):
    """The point-quadrature sum at the points x for each of the inputs (plan precision)."""
    y, w, n = _points(V, T, rule)
    n = n.repeat_interleave(rule, 0)
    lam = torch.as_tensor(_rule(rule)[0], device=DEVICE)
    tri = torch.as_tensor(T, device=DEVICE).long()
    q = []
    for v in inputs:
        v = v.double()
        if case["input"] == "nodal":
            v = torch.einsum("sa,tad->tsd", lam, v[tri]).reshape(-1, 3)
        q.append(w * (v if case["input"] == "sigma" else (v * n).sum(1)))
    return _direct(x, y, torch.stack(q, 1))


def _exact_potential(case, seed):
    X, K = _ball(case["size"])
    bnd = np.sort(np.concatenate([K[:, [1, 2, 3]], K[:, [0, 2, 3]], K[:, [0, 1, 3]], K[:, [0, 1, 2]]]), 1).astype(np.int64)
    opp = np.concatenate([K[:, 0], K[:, 1], K[:, 2], K[:, 3]]).astype(np.int64)
    N = len(X)
    key = (bnd[:, 0] * N + bnd[:, 1]) * N + bnd[:, 2]
    _, first, times = np.unique(key, return_index=True, return_counts=True)
    once = first[times == 1]
    F, O = (torch.as_tensor(a[once], device=DEVICE) for a in (bnd, opp))
    if N * len(F) > TRIANGLE_PAIRS:
        return None
    x = torch.as_tensor(X, device=DEVICE)
    k = torch.as_tensor(K, device=DEVICE).long()
    dt = torch.float64 if case["bits"] == 64 else torch.float32
    m = _field(X, seed).to(dt).double()
    J = x[k[:, 1:]] - x[k[:, :1]]
    vol = torch.linalg.det(J).abs() / 6
    G = torch.linalg.inv(J).transpose(1, 2)  # gradients of the hat functions 1..3
    G = torch.cat([-G.sum(1, keepdim=True), G], 1)
    free = torch.ones(N, dtype=torch.float64, device=DEVICE)
    free[F.reshape(-1)] = 0
    A = torch.einsum("t,tad,tbd->tab", vol, G, G)
    S = torch.sparse_coo_tensor(torch.stack([k.repeat_interleave(4, 1).reshape(-1), k.repeat(1, 4).reshape(-1)]),
                                A.reshape(-1), (N, N)).coalesce()
    diag = torch.zeros(N, dtype=torch.float64, device=DEVICE)
    on = S.indices()[0] == S.indices()[1]
    diag[S.indices()[0][on]] = S.values()[on]
    S = S.to_sparse_csr()
    b = torch.zeros(N, dtype=torch.float64, device=DEVICE)
    b.index_add_(0, k.reshape(-1), (vol[:, None] * torch.einsum("tad,td->ta", G, m[k].mean(1))).reshape(-1))
    b *= free
    phi1, r = torch.zeros_like(b), b.clone()
    z = r * free / diag
    p, rz, stop = z.clone(), r @ z, 1e-13 * float(b.norm())
    for _ in range(5000):
        q = (S @ p) * free
        alpha = rz / (p @ q)
        phi1 += alpha * p
        r -= alpha * q
        if float(r.norm()) <= stop:
            break
        z = r * free / diag
        rz, old = r @ z, rz
        p = z + rz / old * p
    P = x[F]
    n = torch.linalg.cross(P[:, 1] - P[:, 0], P[:, 2] - P[:, 0])
    n = n / n.norm(dim=1, keepdim=True)
    h = ((x[O] - P[:, 0]) * n).sum(1)  # the fourth node lies inside
    flip = (h > 0)[:, None]
    P = torch.where(flip[:, None], P[:, [0, 2, 1]], P)
    n = torch.where(flip, -n, n)
    g = (m[F].mean(1) * n).sum(1) + phi1[O] / h.abs()
    return [phi1 + _triangles(x, P, n, g), phi1]


def exact(case, seed):
    if case["form"] == "potential":
        return _exact_potential(case, seed)
    if case["form"] == "batched":
        parts = _parts(case)
        if sum(len(V) * len(T) * q for V, T, q in parts) > PAIRS:
            return None
        return [_exact_points(case, V, T, q, torch.as_tensor(V, device=DEVICE),
                              [_input(case, V, T, (seed, i, k)) for k in range(case["count"])])
                .reshape(len(V), -1).t().contiguous() for i, (V, T, q) in enumerate(parts)]
    V, T = _surface(case["mesh"], case["size"])
    x = torch.as_tensor(V, device=DEVICE)
    if case["options"] == "triangles":
        if len(V) * len(T) > TRIANGLE_PAIRS:
            return None
        P = x[torch.as_tensor(T, device=DEVICE).long()]
        v = _input(case, V, T, seed).double()
        n = _points(V, T, 1)[2]
        if case["input"] == "nodal":  # the mean of m.n over each triangle
            v = (v[torch.as_tensor(T, device=DEVICE).long()].mean(1) * n).sum(1)
        return _triangles(x, P, n, v)
    probes = torch.as_tensor(_inside(case["mesh"], V, T, case["count"]), device=DEVICE) if case["form"] == "probe" else None
    if (len(V) + (0 if probes is None else len(probes))) * len(T) * case["rule"] > PAIRS:
        return None
    if case["form"] == "states":
        return _exact_points(case, V, T, case["rule"], x,
                             [_input(case, V, T, (seed, k)) for k in range(case["count"])]).reshape(len(V), -1).t().contiguous()
    v = [_input(case, V, T, seed)]
    phi = _exact_points(case, V, T, case["rule"], x, v)
    return phi if probes is None else [phi, _exact_points(case, V, T, case["rule"], probes, v)]
