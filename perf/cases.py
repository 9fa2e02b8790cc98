"""The work whose time matters: the library's calls over the sizes users run them at.

Each case is a dict of plain values: `op` names the entry points, `shape` and `n` the surface (see `surface`), `levels` the
oct-tree, `k0` the wavenumber (rad/m, bodies of 1 to 2 m), `precision` the arithmetic of the problem, `nrhs` the columns.

op            what it stands for
apply         one matrix-vector product y = Z x, the call every Krylov step makes; nrhs columns in one call
adjoint       y = Z^H x, the product of an adjoint solve (gradients of far-field objectives)
near          y = Z_near x, the sparse near part alone (a preconditioner, or an iteration's local part)
farfield      far-zone field of a solution in n_points directions (a bistatic cut)
farfield_adj  the adjoint of that map (the seed of an adjoint solve)
nearfield     scattered field at n_points points off the surface, from currents and charges
setup         a new operator (mesh, tree, near integrals, tables) and its first product
solve         right-hand side of a plane wave, nested solve to 1e-6, far field: a whole scattering run
"""
import functools
import math

import numpy as np
import torch

import paper_1806_04164_gb300 as pg

C0 = 299792458.0
MU0 = 4e-7 * math.pi
EPS0 = 1.0 / (MU0 * C0 * C0)
PRECISIONS = {"fp64": pg.PIE_FP64, "fp32": pg.PIE_FP32, "mixed": pg.PIE_MIXED, "fp32h": pg.PIE_FP32H}
# (tau, kappa a, N_theta): the library's default, and the complex-float point of an inner operator
POINT = {"fp64": (7, 0.08, 8), "mixed": (7, 0.08, 8), "fp32": (3, 0.15, 4), "fp32h": (3, 0.15, 4)}


# ---------------------------------------------------------------- surfaces

def _subdivide(v, f, n):
    """Each triangle into four by its edge midpoints, projected to the unit sphere, n times."""
    for _ in range(n):
        e = np.sort(np.concatenate([f[:, [0, 1]], f[:, [1, 2]], f[:, [2, 0]]]), axis=1)
        e, inv = np.unique(e, axis=0, return_inverse=True)
        m = v[e[:, 0]] + v[e[:, 1]]
        a, b, c = f.T
        ab, bc, ca = len(v) + inv.reshape(3, -1)
        v = np.concatenate([v, m / np.linalg.norm(m, axis=1, keepdims=True)])
        f = np.concatenate([np.stack(t, 1) for t in ((a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca))])
    return v, f


def _outward(v, f):
    nrm = np.cross(v[f[:, 1]] - v[f[:, 0]], v[f[:, 2]] - v[f[:, 0]])
    flip = np.sum(nrm * v[f].sum(1), 1) < 0
    f[flip] = f[flip][:, [0, 2, 1]]
    return f


def _weld(p, f):
    """Points that coincide become one vertex."""
    _, first, inv = np.unique(np.round(p * 1e9).astype(np.int64), axis=0, return_index=True, return_inverse=True)
    return p[first], inv.reshape(-1)[f]


def _grid(n, m):
    i, j = np.meshgrid(np.arange(n), np.arange(m), indexing="ij")
    a = (i * (m + 1) + j).ravel()
    return a, a + m + 1, a + m + 2, a + 1


@functools.lru_cache(maxsize=4)
def surface(shape, n):
    """Vertices and triangles. sphere: icosahedron subdivided n times, R 1 m (20 4^n triangles); ellipsoid: octahedron
    subdivided n times, semi-axes 1, 0.5, 0.5 (8 4^n); cube: side 1 m, n x n squares a face, 4 triangles a square (24 n^2);
    cylinder: R 0.5 m, height 2 m, n segments around, n - 9 rows and n/6 rings a cap; patch: open 0.6 m plate, 2 n^2."""
    if shape == "sphere":
        g = (1 + 5 ** 0.5) / 2
        v = np.array([p for s in (-1, 1) for q in (-g, g) for p in ((0, s, q), (s, q, 0), (q, 0, s))], float)
        d = np.linalg.norm(v[:, None] - v[None], axis=2)
        f = np.array([(i, j, k) for i in range(12) for j in range(i) for k in range(j)
                      if max(d[i, j], d[j, k], d[i, k]) < 2.1])
        v, f = _subdivide(v / np.linalg.norm(v, axis=1, keepdims=True), _outward(v, f), n)
    elif shape == "ellipsoid":
        v = np.concatenate([np.eye(3), -np.eye(3)])
        f = np.array([(x, y, z) for x in (0, 3) for y in (1, 4) for z in (2, 5)])
        v, f = _subdivide(v, _outward(v, f), n)
        v = v * np.array([1.0, 0.5, 0.5])
    elif shape == "cube":
        a, b, c, d = _grid(n, n)
        s = np.linspace(-0.5, 0.5, n + 1)
        u, w = (t.ravel() for t in np.meshgrid(s, s, indexing="ij"))
        q = np.stack([u, w, np.full(u.size, 0.5)], 1)
        mid = len(q) + np.arange(len(a))
        q = np.concatenate([q, (q[a] + q[c]) / 2])
        f = np.concatenate([np.stack(t, 1) for t in ((a, b, mid), (b, c, mid), (c, d, mid), (d, a, mid))])
        faces = [np.roll(q * np.array([1, 1, sg]), r, axis=1) for r in range(3) for sg in (1, -1)]
        v, f = _weld(np.concatenate(faces), np.concatenate([f + len(q) * k for k in range(6)]))
        f = _outward(v, f)
    elif shape == "cylinder":
        rows, rings = n - 9, max(2, n // 6)
        prof = [(r, -1.0) for r in np.linspace(0, 0.5, rings + 1)[:-1]] + [(0.5, z) for z in np.linspace(-1, 1, rows + 1)]
        prof = np.array(prof + [(r, 1.0) for r in np.linspace(0.5, 0, rings + 1)[1:]])
        phi = 2 * np.pi * np.arange(n + 1) / n
        phi[-1] = 0.0
        p = np.stack([prof[:, :1] * np.cos(phi), prof[:, :1] * np.sin(phi), np.repeat(prof[:, 1:], n + 1, 1)], 2).reshape(-1, 3)
        a, b, c, d = _grid(len(prof) - 1, n)
        v, f = _weld(p, np.concatenate([np.stack((a, b, c), 1), np.stack((a, c, d), 1)]))
        f = f[(f[:, 0] != f[:, 1]) & (f[:, 1] != f[:, 2]) & (f[:, 0] != f[:, 2])]
        f = _outward(v, f)
    else:  # patch
        s = np.linspace(-0.3, 0.3, n + 1)
        u, w = (t.ravel() for t in np.meshgrid(s, s, indexing="ij"))
        v = np.stack([u, w, np.zeros(u.size)], 1)
        a, b, c, d = _grid(n, n)
        f = np.stack([np.stack((a, b, c), 1), np.stack((a, c, d), 1)], 1).reshape(-1, 3)
    return np.ascontiguousarray(v), np.ascontiguousarray(f, np.int32)


def triangles(shape, n):
    return {"sphere": 20 * 4 ** n, "ellipsoid": 8 * 4 ** n, "cube": 24 * n * n, "patch": 2 * n * n,
            "cylinder": 2 * n * (n - 9) + n * (4 * max(2, n // 6) - 2)}[shape]


def levels(shape, n):
    """As many as keep the leaf boxes over about 2.5 edges (the library wants 1.5)."""
    side, edge = {"sphere": (2.0, 1.26 / 2 ** n), "ellipsoid": (2.0, 2.2 / 2 ** n), "cube": (1.0, 1.0 / n),
                  "cylinder": (2.0, 3.9 / n), "patch": (0.6, 0.85 / n)}[shape]
    return max(3, 1 + int(math.log2(side / (2.5 * edge))))


# ---------------------------------------------------------------- the cases

def _case(name, op, shape, n, k0, precision, nrhs=1, points=0):
    return {"name": name, "op": op, "shape": shape, "n": n, "levels": levels(shape, n), "k0": k0, "precision": precision,
            "nrhs": nrhs, "points": points}


MHZ100 = 2 * math.pi * 1e8 / C0


def listed():
    return [
        # the smallest problem in use (1280 triangles): a product is launches and latency
        _case("product_1280", "apply", "sphere", 3, 1e-2, "mixed"),
        # the timed workload (819,200 unknowns): one product of a GMRES step
        _case("product_328k", "apply", "sphere", 7, 1e-3, "mixed"),
        # the same product with every part in complex double, the library's default precision
        _case("product_82k_fp64", "apply", "sphere", 6, 1e-3, "fp64"),
        # the inner operator of the nested solve, 20 products per outer step, at the timed workload
        _case("inner_328k", "apply", "sphere", 7, 1e-3, "fp32h"),
        # a batch of excitations on a ragged tree (flat caps, curved side)
        _case("batch8_cylinder", "apply", "cylinder", 128, 1e-2, "mixed", nrhs=8),
        # an adjoint product on the open plate at 100 MHz, an odd grid, all boxes large in wavelengths but the smallest
        _case("adjoint_patch_fp64", "adjoint", "patch", 75, MHZ100, "fp64"),
        # the near part alone, edges and corners in the tree
        _case("near_cube_fp64", "near", "cube", 32, 1e-2, "fp64"),
        # a bistatic cut, its adjoint, and the field on a grid of points near the body
        _case("farfield_181", "farfield", "sphere", 6, 1e-3, "mixed", points=181),
        _case("farfield_adjoint_181", "farfield_adj", "ellipsoid", 6, 1e-2, "mixed", points=181),
        _case("nearfield_1024", "nearfield", "sphere", 5, 1e-2, "mixed", points=1024),
        # a new operator and its first product
        _case("setup_20k", "setup", "sphere", 5, 1e-2, "mixed"),
        # a whole scattering run on a small body
        _case("solve_5k", "solve", "sphere", 4, 1e-2, "mixed", points=181),
    ]


def draw(rng):
    op, precisions, most = rng.choice([
        ("apply", ("mixed", "mixed", "fp64", "fp32h", "fp32"), 330000), ("apply", ("mixed", "mixed", "fp64", "fp32h", "fp32"), 330000),
        ("apply", ("mixed", "fp64", "fp32h"), 50000), ("adjoint", ("fp64", "mixed"), 90000), ("near", ("fp64", "mixed", "fp32h"), 90000),
        ("farfield", ("mixed", "fp64"), 90000), ("farfield_adj", ("mixed", "fp64"), 40000), ("nearfield", ("mixed", "fp64"), 21000),
        ("setup", ("mixed", "fp64", "fp32h"), 30000), ("solve", ("mixed",), 6000)])
    precision = rng.choice(precisions)
    if precision == "fp64":  # a complex double near part costs about four times a float one
        most = min(most, 90000)
    t = math.exp(rng.uniform(math.log(1200), math.log(most)))
    shape = rng.choice(["sphere", "ellipsoid", "cube", "cylinder", "patch"] if op != "solve" else ["sphere", "ellipsoid", "cube"])
    if shape in ("sphere", "ellipsoid"):
        n = max(3, min(7, int(math.log(t / (20 if shape == "sphere" else 8), 4))))
    else:
        n = max(12, int({"cube": (t / 24) ** 0.5, "patch": (t / 2) ** 0.5, "cylinder": 4.5 + (t / 2.67) ** 0.5}[shape]))
        n = n if shape != "cube" else max(7, int((t / 24) ** 0.5))
    k0 = rng.choice([MHZ100, MHZ100 / 100]) if shape == "patch" else 10 ** rng.uniform(-3, -1.5)
    nrhs = rng.choice([1, 1, 1, 2, 3, 5, 8]) if op == "apply" and triangles(shape, n) <= 50000 else 1
    points = rng.randrange(19, 400) if op != "nearfield" else rng.randrange(20, 1100)
    c = _case("", op, shape, n, k0, precision, nrhs, points if op in ("farfield", "farfield_adj", "nearfield", "solve") else 0)
    del c["name"]
    return c


def _problem(case, mesh, precision=None):
    precision = precision or case["precision"]
    tau, kappa_a, ntheta = POINT[precision]
    return pg.Problem(mesh, case["k0"], case["levels"], root_side=2.0 if case["shape"] == "sphere" else 0.0, tau=tau,
                      kappa_a=kappa_a, ntheta=ntheta, precision=PRECISIONS[precision], max_nrhs=case["nrhs"])


def _normal(shape, gen, dtype=torch.complex128):
    """Complex normal entries, real and imaginary parts N(0, 1)."""
    return (torch.randn(shape, generator=gen, device="cuda", dtype=torch.complex128) * 2 ** 0.5).to(dtype)


def _directions(n, seed):
    """A cut through the body: n directions over 180 degrees in a plane that the seed turns."""
    th, ph = np.linspace(0, np.pi, n), 0.37 * (seed % 17)
    return np.stack([np.sin(th) * np.cos(ph), np.sin(th) * np.sin(ph), np.cos(th)], 1)


def _wave(seed):
    r = np.random.RandomState(seed % 2 ** 31)
    k, e = r.randn(3), r.randn(3)
    k /= np.linalg.norm(k)
    e -= k * (k @ e)
    return k, e / np.linalg.norm(e)


def _points(case, seed):
    """Points off the surface: on a shell 1.3 to 2.5 times the body's half diagonal."""
    r = np.random.RandomState(seed % 2 ** 31)
    p = r.randn(case["points"], 3)
    half = np.linalg.norm(np.abs(surface(case["shape"], case["n"])[0]).max(0))
    return p / np.linalg.norm(p, axis=1, keepdims=True) * half * r.uniform(1.3, 2.5, (len(p), 1))


def _inputs(case, seed, N, T):
    """The call's arguments beside the operator, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    op, n = case["op"], case["points"]
    f32 = case["precision"] in ("fp32", "fp32h")
    s = {}
    if op in ("apply", "adjoint", "near", "setup"):
        s["x"] = _normal((case["nrhs"], N) if case["nrhs"] > 1 else (N,), gen, torch.complex64 if f32 else torch.complex128)
    if op in ("farfield", "nearfield"):
        s["x"] = _normal((N,), gen)
    if op in ("farfield", "farfield_adj", "solve"):
        s["dirs"] = _directions(n, seed)
    if op == "farfield_adj":
        s["E"] = _normal((n, 3), gen)
    if op == "nearfield":
        s["rho"], s["pts"] = _normal((T,), gen) * EPS0, _points(case, seed)
    if op == "solve":
        s["wave"] = _wave(seed)
    return s


def prepare(case, seed):
    xyz, tri = surface(case["shape"], case["n"])
    if case["op"] == "setup":
        T = len(tri)
        edges = 3 * T // 2 if case["shape"] != "patch" else 3 * case["n"] ** 2 - 2 * case["n"]
        return {"case": case, "xyz": xyz, "tri": tri, **_inputs(case, seed, edges + T, T)}
    mesh = pg.Mesh(xyz, tri)
    s = {"case": case, "pr": _problem(case, mesh)}
    if case["op"] == "solve":
        s["inner"] = _problem(case, mesh, "fp32h")
    return {**s, **_inputs(case, seed, s["pr"].N, s["pr"].T)}


def run(s):
    op = s["case"]["op"]
    if op == "apply":
        return s["pr"].apply(s["x"])
    if op == "adjoint":
        return s["pr"].apply_t(s["x"], conj=True)
    if op == "near":
        return s["pr"].apply(s["x"], near_only=True)
    if op == "farfield":
        return s["pr"].farfield(s["x"], s["dirs"])
    if op == "farfield_adj":
        return s["pr"].farfield_adjoint(s["E"], s["dirs"])
    if op == "nearfield":
        return s["pr"].nearfield(s["x"], s["rho"], s["pts"])
    if op == "setup":
        return _problem(s["case"], pg.Mesh(s["xyz"], s["tri"])).apply(s["x"])
    b = s["pr"].rhs_planewave(*s["wave"])
    x, _ = s["pr"].solve_nested(b, s["inner"])
    return {"x": x, "E": s["pr"].farfield(x, s["dirs"])}


# ---------------------------------------------------------------- what a pass cannot do without

def _side(shape, v):
    return 2.0 if shape == "sphere" else float((v.max(0) - v.min(0)).max())


def _leaf(v, f, side, nlev):
    """Leaf box of every triangle, by its centroid."""
    x0, nl = (v.max(0) + v.min(0)) * 0.5 - side * 0.5, 2 ** (nlev - 1)
    cent = ((v[f[:, 0]] + v[f[:, 1]]) + v[f[:, 2]]) / 3.0
    return np.clip(np.floor((cent - x0) * (nl / side)).astype(np.int64), 0, nl - 1)


@functools.lru_cache(maxsize=32)
def _counts(shape, n, nlev):
    """Triangles, unknowns, near pairs, and per level 3..L boxes and interaction pairs of the one-box-buffer tree."""
    v, f = surface(shape, n)
    leaf = _leaf(v, f, _side(shape, v), nlev)
    step = np.array([(i, j, k) for i in (-1, 0, 1) for j in (-1, 0, 1) for k in (-1, 0, 1)])
    code = lambda c: ((c[..., 0] + 2) * 4096 + c[..., 1] + 2) * 4096 + c[..., 2] + 2  # noqa: E731

    def near(count, keys):
        """Pairs of neighbouring boxes, each box counted `count` times."""
        at = np.searchsorted(keys, code(cells[:, None] + step).clip(0, keys[-1]))
        hit = keys[at] == code(cells[:, None] + step)
        return int((count[:, None] * np.where(hit, count[at], 0)).sum())

    per_level, pairs = [], 0
    for lev in range(nlev, 1, -1):
        cells, cnt = np.unique(leaf >> (nlev - lev), axis=0, return_counts=True)
        order = np.argsort(code(cells))
        cells, cnt = cells[order], cnt[order]
        keys = code(cells)
        if lev == nlev:
            pairs = near(cnt, keys)
        # boxes, pairs of neighbours, and children of neighbours' pairs (the level below)
        kids = np.unique(leaf >> (nlev - lev - 1), axis=0)[:, :] >> 1 if lev < nlev else cells
        kid_count = np.zeros(len(keys), np.int64)
        np.add.at(kid_count, np.searchsorted(keys, code(kids)), 1)
        per_level.append((lev, len(cells), near(np.ones(len(cells), np.int64), keys), near(kid_count, keys)))
    per_level.sort()
    lists = [(b, per_level[i][3] - own) for i, (lev, b, own, _) in enumerate(per_level[1:])]
    T = len(f)
    E = 3 * T // 2 if shape != "patch" else 3 * n * n - 2 * n
    return T, E + T, pairs, lists


def _product(case, precision, nrhs, far=True):
    """Bytes and operations of products of nrhs columns: near moments and tables read once, vectors read and written."""
    T, N, pairs, lists = _counts(case["shape"], case["n"], case["levels"])
    P = 2 * POINT[precision][2] ** 2
    moment = {"fp64": 16, "mixed": 8, "fp32": 8, "fp32h": 4}[precision]
    c = 16 if precision in ("fp64", "mixed") else 8
    by, fl = 8 * moment * pairs + 2 * c * N * nrhs, 96 * pairs * nrhs
    if far:
        # radiation tables of half the samples (their antipodes are conjugates), 4 a triangle; 5 densities a box
        by += 4 * T * P // 2 * c
        fl += nrhs * (2 * 64 * T * P // 2 + sum(40 * il * P for _, il in lists) + sum(2 * 5 * 40 * P * b for b, _ in lists[1:]))
    return by, fl


def work(case):
    T, N, pairs, _ = _counts(case["shape"], case["n"], case["levels"])
    op, p = case["op"], case["points"]
    if op in ("apply", "adjoint", "near"):
        by, fl = _product(case, case["precision"], case["nrhs"], op != "near")
    elif op in ("farfield", "farfield_adj"):  # 7 points a triangle and direction: a phase and a vector sum
        by, fl = 16 * N + 48 * p + 72 * T, 7 * T * p * 40
    elif op == "nearfield":
        by, fl = 16 * (N + T) + 72 * p + 72 * T, 7 * T * p * 60
    elif op == "setup":  # 49 point pairs a near pair, both orders at once; moments written, then read by the product
        by, fl = _product(case, case["precision"], 1)
        by, fl = by + 8 * {"fp64": 16, "mixed": 8, "fp32h": 4}[case["precision"]] * pairs, fl + 49 * 30 * pairs // 2
    else:  # a run of about 300 inner and 30 outer products
        bo, fo = _product(case, "mixed", 1)
        bi, fi = _product(case, "fp32h", 1)
        by, fl = 30 * bo + 300 * bi, 30 * fo + 300 * fi
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------- the same results in 64 bits

class _Geometry:
    """Mesh tables on the GPU in double: RWG functions on interior edges sorted by (min, max) vertex, then pulses."""

    def __init__(self, case):
        v, f = surface(case["shape"], case["n"])
        T = len(f)
        e = np.stack([f, np.roll(f, -1, 1)], 2).reshape(-1, 2).astype(np.int64)
        key = np.minimum(e[:, 0], e[:, 1]) * len(v) + np.maximum(e[:, 0], e[:, 1])
        uniq, inv, cnt = np.unique(key, return_inverse=True, return_counts=True)
        number = np.where(cnt == 2, np.cumsum(cnt == 2) - 1, -1)[inv.reshape(-1)].reshape(T, 3)
        sign = np.where(e[:, 0] < e[:, 1], 1.0, -1.0).reshape(T, 3)
        on = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
        self.v = on(v[f])
        self.cent = self.v.sum(1) / 3
        cr = torch.linalg.cross(self.v[:, 1] - self.v[:, 0], self.v[:, 2] - self.v[:, 0])
        self.area = cr.norm(dim=1) / 2
        length = (self.v - self.v.roll(-1, 1)).norm(dim=2)
        self.h2 = (length ** 2).max(1).values
        self.edge, self.E, self.T = on(np.maximum(number, 0)), int((cnt == 2).sum()), T
        self.c = on(np.where(number >= 0, sign, 0.0)) * length / (2 * self.area[:, None])
        self.dcp = self.cent[:, None] - self.v.roll(1, 1)  # the free vertex of edge (k, k + 1) is k + 2
        s15 = 15 ** 0.5
        rule = [(1 / 3, 1 / 3, 1 / 3, 9 / 40)]
        for a, w in (((6 - s15) / 21, (155 - s15) / 1200), ((6 + s15) / 21, (155 + s15) / 1200)):
            rule += [(1 - 2 * a, a, a, w), (a, 1 - 2 * a, a, w), (a, a, 1 - 2 * a, w)]
        rule = on(np.array(rule))
        self.q = torch.einsum("jk,tkd->tjd", rule[:, :3], self.v)  # [T, 7, 3]
        self.w = rule[:, 3] * self.area[:, None]
        self.u = self.q - self.cent[:, None]
        x, w = np.polynomial.legendre.leggauss(8)
        x, w = (x + 1) / 2, w / 2
        a, b = np.repeat(x, 8), np.tile(x, 8) * (1 - np.repeat(x, 8))
        self.rule64 = on(np.stack([1 - a - b, a, b, 2 * np.repeat(w, 8) * np.tile(w, 8) * (1 - a)], 1))

    def local(self, x, k0):
        """[T, 6] densities of each triangle: J = a (r - c) + beta, sigma, d = 2 a + w^2 eps0 sigma."""
        xe, s = x[self.edge] * self.c, x[self.E:]
        a = xe.sum(1)
        return torch.cat([a[:, None], (xe[:, :, None] * self.dcp).sum(1), s[:, None], (2 * a + (k0 * C0) ** 2 * EPS0 * s)[:, None]], 1)

    def test(self, pot):
        """Galerkin testing of [T, 6] potentials (U, V, T1, T2)."""
        edge = self.c * (pot[:, :1] + (self.dcp * pot[:, None, 1:4]).sum(2) + 2 * pot[:, 4:5])
        y = torch.zeros(self.E, dtype=pot.dtype, device=pot.device).index_add_(0, self.edge.reshape(-1), edge.reshape(-1))
        return torch.cat([y, pot[:, 5]])

    def current(self, loc):
        return loc[:, :1, None] * self.u + loc[:, None, 1:4]  # [T, 7, 3]


def _static(r, v):
    """int 1/R and int (r' - r)/R over flat triangles v [n, 3, 3] at points r [n, p, 3] (Wilton et al. 1984)."""
    nrm = torch.linalg.cross(v[:, 1] - v[:, 0], v[:, 2] - v[:, 0])
    nrm = (nrm / nrm.norm(dim=1, keepdim=True))[:, None]
    d = ((r - v[:, None, 0]) * nrm).sum(2)
    one, vec = torch.zeros_like(d), torch.zeros_like(r)
    for k in range(3):
        a, b = v[:, None, k], v[:, None, (k + 1) % 3]
        s = (b - a) / (b - a).norm(dim=2, keepdim=True)
        m = torch.linalg.cross(s, nrm)
        lp, lm, p0 = ((b - r) * s).sum(2), ((a - r) * s).sum(2), ((a - r) * m).sum(2)
        rp, rm, r2 = (r - b).norm(dim=2), (r - a).norm(dim=2), p0 * p0 + d * d
        f = torch.where(lm >= 0, (rp + lp) / (rm + lm), torch.where(lp <= 0, (rm - lm) / (rp - lp), (rp + lp) * (rm - lm) / r2)).log()
        f = torch.where(r2 > 1e-24 * ((b - a) ** 2).sum(2), f, 0.0)
        at = torch.atan(p0 * lp / (r2 + d.abs() * rp)) - torch.atan(p0 * lm / (r2 + d.abs() * rm))
        one += p0 * f - d.abs() * torch.nan_to_num(at)
        vec += 0.5 * (r2 * f + lp * rp - lm * rm)[..., None] * m
    return one, vec - (d * one)[..., None] * nrm


def _singular(g, t, s, k0):
    """[n, 8] moments of near-singular pairs, test t, source s: static part in closed form, the rest by the 7-point rule."""
    r = torch.einsum("jk,tkd->tjd", g.rule64[:, :3], g.v[t])
    w = g.rule64[:, 3] * g.area[t][:, None]
    one, vec = _static(r, g.v[s])
    K = (one / (4 * math.pi)).to(torch.complex128)
    K1 = ((vec + (r - g.cent[s][:, None]) * one[..., None]) / (4 * math.pi)).to(torch.complex128)
    for j in range(7):
        R = (r - g.q[s][:, None, j]).norm(dim=2)
        rem = torch.where(R > 0, torch.polar(2 * torch.sin(k0 * R / 2) / (4 * math.pi * R), k0 * R / 2) * 1j, 1j * k0 / (4 * math.pi))
        rem = rem * g.w[s][:, None, j]
        K += rem
        K1 += rem[..., None] * g.u[s][:, None, j]
    u, wK = r - g.cent[t][:, None], w * K
    return torch.cat([wK.sum(1, True), (wK[..., None] * u).sum(1), (w[..., None] * K1).sum(1), (w[..., None] * u * K1).sum((1, 2))[:, None]], 1)


def _moments(g, rows, k0):
    """[8, rows, T] pair moments of test triangles `rows` against all: m0, mt, ms, mts."""
    m = torch.zeros((8, len(rows), g.T), dtype=torch.complex128, device="cuda")
    for i in range(7):
        K = torch.zeros((4, len(rows), g.T), dtype=torch.complex128, device="cuda")
        for j in range(7):
            R = (g.q[rows, i][:, None] - g.q[None, :, j]).norm(dim=2)
            G = torch.polar(g.w[:, j] / (4 * math.pi * R.clamp_min(1e-300)), k0 * R)
            K[0] += G
            for d in range(3):
                K[1 + d] += G * g.u[:, j, d]
        w, u = g.w[rows, i][:, None], g.u[rows, i]
        m[0] += w * K[0]
        for d in range(3):
            ud = w * u[:, d:d + 1]
            m[1 + d] += ud * K[0]
            m[4 + d] += w * K[1 + d]
            m[7] += ud * K[1 + d]
    d2 = ((g.cent[rows][:, None] - g.cent[None]) ** 2).sum(2)
    t, s = torch.nonzero(d2 < 2.25 * torch.maximum(g.h2[rows][:, None], g.h2[None]), as_tuple=True)
    for a in range(0, len(t), 20000):
        ti, si = t[a:a + 20000], s[a:a + 20000]
        x, y = _singular(g, rows[ti], si, k0), _singular(g, si, rows[ti], k0)
        m[:, ti, si] = (0.5 * (x + y[:, [0, 4, 5, 6, 1, 2, 3, 7]])).T
    return m


def _potentials(m, loc):
    """[rows, 6] potentials of moments m [8, rows, T] and densities loc [T, 6]."""
    p = torch.empty((m.shape[1], 6), dtype=torch.complex128, device="cuda")
    p[:, 0] = m[7] @ loc[:, 0] + m[1] @ loc[:, 1] + m[2] @ loc[:, 2] + m[3] @ loc[:, 3]
    for d in range(3):
        p[:, 1 + d] = m[4 + d] @ loc[:, 0] + m[0] @ loc[:, 1 + d]
    p[:, :4] *= MU0
    p[:, 4:] = m[0] @ loc[:, 4:]
    return p


def _chunks(g, size):
    return torch.arange(g.T, device="cuda").split(max(1, size // g.T))


def _farfield(g, case, x, dirs):
    J = g.current(g.local(x, case["k0"])) * g.w[..., None]
    F = torch.stack([(torch.polar(torch.ones_like(g.w), -case["k0"] * (g.q @ r))[..., None] * J).sum((0, 1)) for r in dirs])
    return 1j * case["k0"] * C0 * MU0 / (4 * math.pi) * (F - dirs * (F * dirs).sum(1, keepdim=True))


def _farfield_adjoint(g, case, E, dirs):
    E = (E - dirs * (E * dirs).sum(1, keepdim=True)) * (-1j * case["k0"] * C0 * MU0 / (4 * math.pi))
    h = sum(torch.polar(torch.ones_like(g.w), case["k0"] * (g.q @ r))[..., None] * e for r, e in zip(dirs, E)) * g.w[..., None]
    pot = torch.zeros((g.T, 6), dtype=torch.complex128, device="cuda")
    pot[:, 0], pot[:, 1:4] = (h * g.u).sum((1, 2)), h.sum(1)
    return g.test(pot)


def _nearfield(g, case, x, rho, pts):
    k0, J = case["k0"], g.current(g.local(x, case["k0"]))
    out = []
    for p in pts:
        d = p - g.q
        R = d.norm(dim=2)
        G = torch.polar(g.w / (4 * math.pi * R), k0 * R)
        out.append(1j * k0 * C0 * MU0 * (G[..., None] * J).sum((0, 1))
                   - ((rho[:, None] * G * (1j * k0 - 1 / R) / R)[..., None] * d).sum((0, 1)) / EPS0)
    return torch.stack(out)


def _solution(g, case, wave, tol=1e-9):
    """The plane wave's solution with the dense operator: GMRES without restart, scaled by the diagonal's magnitude."""
    k, e = (torch.from_numpy(a).cuda() for a in wave)
    er = g.q @ e
    phi = -er * torch.polar(torch.ones_like(er), case["k0"] * (g.q @ k)) * g.w
    pot = torch.zeros((g.T, 6), dtype=torch.complex128, device="cuda")
    pot[:, 0] = -(phi[..., None] * g.u * k).sum((1, 2)) / C0
    pot[:, 1:4] = -phi.sum(1, keepdim=True) * k / C0
    pot[:, 5] = -1j * case["k0"] * C0 * EPS0 * phi.sum(1)
    b = g.test(pot)
    m = [_moments(g, rows, case["k0"]) for rows in _chunks(g, 1 << 23)]
    product = lambda x: g.test(torch.cat([_potentials(c, g.local(x, case["k0"])) for c in m]))  # noqa: E731
    # any positive scaling does here: the pulse block against the RWG block, by their self terms
    own = torch.cat([c[:, torch.arange(c.shape[1], device="cuda"), rows] for c, rows in zip(m, _chunks(g, 1 << 23))], 1)[0].abs()
    edge = torch.zeros(g.E, dtype=torch.float64, device="cuda").index_add_(
        0, g.edge.reshape(-1), (MU0 * own[:, None] * (g.c * g.dcp.norm(dim=2)) ** 2).reshape(-1))
    D = torch.cat([edge, (case["k0"] * C0) ** 2 * EPS0 * own]) ** -0.5
    V, H = [D * b / (D * b).norm()], torch.zeros((901, 900), dtype=torch.complex128, device="cuda")
    rhs = torch.zeros(901, 1, dtype=torch.complex128, device="cuda")
    rhs[0] = (D * b).norm()
    for j in range(900):
        w, B = D * product(D * V[j]), torch.stack(V)
        for _ in range(2):
            h = B.conj() @ w
            w, H[:j + 1, j] = w - h @ B, H[:j + 1, j] + h
        H[j + 1, j] = w.norm()
        V.append(w / H[j + 1, j])
        if j % 20 == 19:
            y = torch.linalg.lstsq(H[:j + 2, :j + 1], rhs[:j + 2]).solution
            if (H[:j + 2, :j + 1] @ y - rhs[:j + 2]).norm() < tol * rhs.norm():
                break
    return D * (y[:, 0] @ torch.stack(V[:len(y)]))


def exact(case, seed):
    """Direct sums over all triangles; None where the dense operator would take too long."""
    op, k0 = case["op"], case["k0"]
    T = triangles(case["shape"], case["n"])
    if T > {"apply": 21000, "adjoint": 21000, "setup": 21000, "near": 25000, "solve": 6000}.get(op, 10 ** 6):
        return None
    g = _Geometry(case)
    s = _inputs(case, seed, g.E + g.T, g.T)
    if "dirs" in s:
        dirs = torch.from_numpy(s["dirs"]).cuda()
    if op == "farfield":
        return _farfield(g, case, s["x"], dirs)
    if op == "farfield_adj":
        return _farfield_adjoint(g, case, s["E"], dirs)
    if op == "nearfield":
        return _nearfield(g, case, s["x"], s["rho"], torch.from_numpy(s["pts"]).cuda())
    if op == "solve":
        x = _solution(g, case, s["wave"])
        return {"x": x, "E": _farfield(g, case, x, dirs)}
    x = s["x"].to(torch.complex128).reshape(-1, g.E + g.T)
    x = x.conj().resolve_conj() if op == "adjoint" else x  # Z^H x = conj(Z conj x), Z being symmetric
    if op == "near":
        v, f = surface(case["shape"], case["n"])
        leaf = torch.from_numpy(_leaf(v, f, _side(case["shape"], v), case["levels"])).cuda()
    loc = [g.local(c, k0) for c in x]
    pot = [[] for _ in loc]
    for rows in _chunks(g, 1 << 23):
        m = _moments(g, rows, k0)
        if op == "near":
            m *= ((leaf[rows][:, None] - leaf[None]).abs().amax(2) <= 1)
        for p, c in zip(pot, loc):
            p.append(_potentials(m, c))
    y = torch.stack([g.test(torch.cat(p)) for p in pot])
    y = y.conj().resolve_conj() if op == "adjoint" else y
    return y.reshape(s["x"].shape)
