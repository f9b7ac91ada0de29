"""Measured cases of the radiative-transfer library: what its users have it do, through the public API.

Kinds of case
  apply   rt_apply on an operator that the caller keeps (every iteration of a caller's own solver)
  solve   the whole call for a new problem: rt_build_operator, rt_solve_fixed_point, free
  source  rt_build_source_operator + rt_apply_source on a kept operator (new emitter coefficients)
  batch   rt_build_batch + rt_solve_batch on a list of independent instances
  serve   a burst of requests through a running Server

Geometry: Kuhn meshes of the unit cube (n vertices per axis) or of the box-minus-cube domain, the
inner vertices moved by a seeded fraction of the cell, as an unstructured mesh has them.  The
absorption amplitude, the wall's reflection coefficient and every vector come from the seed too.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

import paper_2306_05789_gb300 as rt

SIGMA = math.pi ** 4 / 15.0
TERMS_FLOPS = 60          # arithmetic of one kernel value (distance, optical depth, exponential)


# ------------------------------------------------------------------ the cases
def _case(name, kind, **kw):
    c = dict(name=name, kind=kind, geometry="cube", n=0, F=1, shared=False, grey=False, mode="hmatrix", prec="f32",
             refine=False, bins=0, count=0, tol=1e-6)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest call: one matvec of the plain dense FP64 method (12^3, grey, one channel)
        _case("apply_dense12_f64", "apply", n=12, grey=True, mode="dense", prec="f64"),
        # a small multi-frequency operator of odd channel count: launch latency and ragged leaves
        _case("apply_n19_F5", "apply", n=19, F=5),
        # the headline operator's matvec: 32^3, 16 channels, FP32
        _case("apply_n32_F16", "apply", n=32, F=16),
        # 64 channels sharing kappa, BF16 far field: the multi-right-hand-side matvec
        _case("apply_n40_F64s_bf16", "apply", n=40, F=64, shared=True, prec="bf16"),
        # the plain method end to end: dense FP64, grey, iterated to 1e-10
        _case("solve_dense12_f64", "solve", n=12, grey=True, mode="dense", prec="f64", tol=1e-10),
        # a small problem end to end (odd size): host path and launches beside the kernels
        _case("solve_n13_F3", "solve", n=13, F=3),
        # the headline workload end to end: 32^3, 16 channels and 16 operators, FP32
        _case("solve_n32_F16", "solve", n=32, F=16),
        # the shared-kappa workload end to end: one operator, 64 channels, BF16 far field with refinement
        _case("solve_n41_F64s_bf16", "solve", n=41, F=64, shared=True, prec="bf16", refine=True),
        # box minus cube: gridded kappa, opaque box, three walls and their corner paths
        _case("solve_box15", "solve", geometry="box", n=15, grey=True),
        # the surface-to-volume matrix for new emitter coefficients, 32^3, 8 channels
        _case("source_n32_F8", "source", n=32, F=8),
        # independent instances of 8..24 vertices per axis and 1..8 channels, solved together
        _case("batch_20", "batch", n=24, F=8, count=20),
        # a burst of requests on a running server, BF16 far field with refinement
        _case("serve_5", "serve", n=28, F=16, count=5, prec="bf16", refine=True),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo - 0.49), math.log(hi + 0.49)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "solve", "solve", "source", "batch", "serve"])
    if kind == "apply":
        form = rng.choice(["dense", "groups", "groups", "shared"])
        if form == "dense":
            return _draw("apply", n=rng.randint(6, 15), F=rng.randint(1, 3), mode="dense",
                         prec=rng.choice(["f64", "f32"]))
        if form == "shared":
            return _draw("apply", n=_log_int(rng, 16, 38), F=16 * rng.randint(1, 4), shared=True,
                         prec=rng.choice(["bf16", "f16", "f32"]), refine=rng.random() < 0.3)
        return _draw("apply", n=_log_int(rng, 9, 31), F=_log_int(rng, 1, 16), prec=rng.choice(["f32", "f32", "bf16", "f16"]))
    if kind == "solve":
        form = rng.choice(["groups", "groups", "shared", "binned", "box", "dense"])
        if form == "box":
            return _draw("solve", geometry="box", n=10, F=rng.randint(1, 12))
        if form == "dense":
            return _draw("solve", n=rng.randint(6, 12), F=rng.randint(1, 3), mode="dense", prec="f64", tol=1e-10)
        if form == "shared":
            return _draw("solve", n=_log_int(rng, 12, 38), F=_log_int(rng, 2, 64), shared=True,
                         prec=rng.choice(["f32", "bf16", "f16"]), refine=True)
        if form == "binned":
            return _draw("solve", n=_log_int(rng, 10, 30), F=_log_int(rng, 8, 24), bins=rng.randint(2, 8))
        return _draw("solve", n=_log_int(rng, 8, 30), F=_log_int(rng, 1, 16))
    if kind == "source":
        return _draw("source", n=_log_int(rng, 10, 32), F=_log_int(rng, 1, 8))
    if kind == "batch":
        return _draw("batch", n=rng.randint(10, 22), F=rng.randint(1, 8), count=rng.randint(2, 18))
    return _draw("serve", n=rng.randint(17, 26), F=_log_int(rng, 1, 16), count=rng.randint(1, 5),
                 prec=rng.choice(["bf16", "f32"]), refine=True)


def _draw(kind, **kw):
    c = _case("", kind, **kw)
    del c["name"]
    return c


# ------------------------------------------------------------------- problems
_KUHN = ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0))


def _grid_mesh(dims, h, rng, hole=0):
    """Kuhn mesh of dims cells of size h; hole: the cells below that index on every axis are left out.
    Inner vertices are moved by up to 0.12 h per axis."""
    vx, vy, vz = (d + 1 for d in dims)
    k, j, i = np.meshgrid(np.arange(vz), np.arange(vy), np.arange(vx), indexing="ij")
    ijk = np.stack([i.ravel(), j.ravel(), k.ravel()], axis=1)
    ck, cj, ci = (a.ravel() for a in np.meshgrid(*(np.arange(d) for d in dims[::-1]), indexing="ij"))
    keep = (ci >= hole) | (cj >= hole) | (ck >= hole)
    cell = np.stack([ci, cj, ck], axis=1)[keep]
    tets = []
    for p in _KUHN:
        corner = [cell]
        for a in p:
            nxt = corner[-1].copy()
            nxt[:, a] += 1
            corner.append(nxt)
        tets.append(np.stack([c[:, 0] + vx * (c[:, 1] + vy * c[:, 2]) for c in corner], axis=1))
    tet = np.stack(tets, axis=1).reshape(-1, 4)
    inner = ((ijk > 0) & (ijk < np.array(dims))).all(axis=1) & ~(ijk <= hole).all(axis=1)
    xyz = ijk * float(h)
    xyz[inner] += rng.uniform(-0.12 * h, 0.12 * h, size=(int(inner.sum()), 3))
    used = np.zeros(len(xyz), dtype=bool)
    used[tet.ravel()] = True
    new_id = np.cumsum(used) - 1
    return xyz[used], new_id[tet].astype(np.int32), new_id


def _face_triangles(n):
    """Triangles of the face x = 0 of the n^3 cube mesh, outward (-x) normal."""
    kk, jj = (a.ravel() for a in np.meshgrid(np.arange(n - 1), np.arange(n - 1), indexing="ij"))
    a, b = n * jj + n * n * kk, n * (jj + 1) + n * n * kk
    c, d = n * (jj + 1) + n * n * (kk + 1), n * jj + n * n * (kk + 1)
    return np.stack([np.stack([a, c, b], axis=1), np.stack([a, d, c], axis=1)], axis=1).reshape(-1, 3).astype(np.int32)


def _freqs(F, shared, grey):
    if grey:
        one = np.ones(1)
        return SimpleNamespace(F=1, nu=one, w=one, c=one, albedo=np.zeros(1), group=None)
    d = 1.9 / F
    nu = 0.1 + (np.arange(F) + 0.5) * d
    return SimpleNamespace(F=F, nu=nu, w=np.full(F, d), c=np.ones(F) if shared else 0.5 + nu,
                           albedo=np.full(F, 0.3), group=None)


def _problem(xyz, tet, tri, kappa, wall, freqs, grey, Q0=1.0, **more):
    return SimpleNamespace(xyz=xyz, tet=tet, emit_tri=tri, kappa=kappa, wall=wall, freqs=freqs, grey=grey, Q0=Q0,
                           T_emit=1.0, N=xyz.shape[0], **more)


def _wall(normal, R0):
    return SimpleNamespace(p=(0.0, 0.0, 0.0), n=normal, R0=R0)


def _cube(n, F, shared, grey, rng):
    xyz, tet, _ = _grid_mesh((n - 1,) * 3, 1.0 / (n - 1), rng)
    if grey:
        kappa = SimpleNamespace(kind=rt.RT_KAPPA_CONST, k0=1.0, amp=0.0)
    else:
        kappa = SimpleNamespace(kind=rt.RT_KAPPA_SINPROD, k0=1.0, amp=float(rng.uniform(0.2, 0.8)))
    return _problem(xyz, tet, _face_triangles(n), kappa, _wall((0.0, 0.0, -1.0), float(rng.uniform(0.2, 0.8))),
                    _freqs(F, shared, grey), grey)


def _box(n, F, grey, rng):
    """(0, 0.6) x (0, 1) x (0, 0.6) in cells of 1/n (n a multiple of 5) minus an opaque emitting cube at
    the origin, of the whole cells that 0.1 needs."""
    dims, h = (3 * n // 5, n, 3 * n // 5), 1.0 / n
    m = -(-n // 10)
    xyz, tet, new_id = _grid_mesh(dims, h, rng, hole=m)
    vx, vy = dims[0] + 1, dims[1] + 1
    tri = []
    for axis in range(3):   # the cube's faces inside the domain, normals pointing into the cube
        u, v = [d for d in range(3) if d != axis]
        for a in range(m):
            for b in range(m):
                q = []
                for da, db in ((0, 0), (1, 0), (1, 1), (0, 1)):
                    p = [0, 0, 0]
                    p[axis], p[u], p[v] = m, a + da, b + db
                    q.append(int(new_id[p[0] + vx * (p[1] + vy * p[2])]))
                for t in ((q[0], q[1], q[2]), (q[0], q[2], q[3])):
                    e = np.cross(xyz[t[1]] - xyz[t[0]], xyz[t[2]] - xyz[t[0]])
                    tri.append(t if e[axis] < 0 else (t[0], t[2], t[1]))
    grid = 10.0 * rng.uniform(0.9, 1.1, size=(6, 10, 6))
    grid[0, 1:, 0] *= 1e-3   # the duct that prolongs the cube
    kappa = SimpleNamespace(kind=rt.RT_KAPPA_GRID, k0=0.0, amp=0.0, grid=grid.astype(np.float32),
                            bbox=(0.0, 0.0, 0.0, 0.6, 1.0, 0.6))
    walls = [_wall(tuple(-1.0 if d == a else 0.0 for d in range(3)), 1.0) for a in range(3)]
    return _problem(xyz, tet, np.array(tri, dtype=np.int32), kappa, walls[0], _freqs(F, False, grey), grey, Q0=0.1,
                    more_walls=tuple(walls[1:]), corner=True,
                    obstacles=(SimpleNamespace(lo=(0.0, 0.0, 0.0), hi=(m * h, m * h, m * h)),))


def _one(case, seed):
    rng = np.random.default_rng(seed)
    if case["geometry"] == "box":
        return _box(case["n"], case["F"], case["grey"], rng)
    return _cube(case["n"], case["F"], case["shared"], case["grey"], rng)


def _sizes(case):
    """(n, F) of the instances of a batch or of a burst: spread over the range, the same for every seed."""
    rng = np.random.default_rng(100 * case["count"] + case["n"])
    lo = 8 if case["kind"] == "batch" else 16
    return [(int(rng.integers(lo, case["n"] + 1)), int(rng.integers(1, case["F"] + 1))) for _ in range(case["count"])]


def _many(case, seed):
    rng = np.random.default_rng(seed)
    return [_cube(n, F, False, False, rng) for n, F in _sizes(case)]


def _hparams(case):
    if case["mode"] == "dense":
        return rt.hparams(mode=rt.RT_MODE_DENSE, prec=rt.RT_PREC_F64 if case["prec"] == "f64" else rt.RT_PREC_F32)
    far = {"f32": rt.RT_PREC_F32, "bf16": rt.RT_PREC_BF16, "f16": rt.RT_PREC_F16}[case["prec"]]
    return rt.hparams(far_prec=far, refine=1 if case["refine"] and case["prec"] != "f32" else 0,
                      kappa_bins=case["bins"])


def _refine_tol(case):
    return 1e-3 if case["refine"] and case["prec"] != "f32" else 0.0


def _vector_type(case):
    return torch.float64 if case["mode"] == "dense" and case["prec"] == "f64" else torch.float32


def _emitter_vertices(p):
    return np.unique(p.emit_tri)


def _random(shape, seed, dtype):
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    return torch.rand(shape, generator=gen, device="cuda", dtype=dtype)


# -------------------------------------------------------------- prepare / run
def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return dict(case=case, problems=_many(case, seed), hp=_hparams(case))
    if kind == "serve":
        srv = rt.Server(_hparams(case), slots=4, tol=case["tol"], refine_tol=_refine_tol(case))
        return dict(case=case, problems=_many(case, seed), server=srv)
    p = _one(case, seed)
    st = dict(case=case, problem=p, hp=_hparams(case))
    F, N, vt = p.freqs.F, p.N, _vector_type(case)
    if kind == "solve":
        st["J"] = torch.zeros(F, N, dtype=vt, device="cuda")
        st["T"] = torch.zeros(N, dtype=torch.float64, device="cuda")
        return st
    st["op"] = rt.rt_build_operator(p, st["hp"])
    if kind == "apply":
        st["X"] = _random((F, N), seed, vt)
        st["Y"] = torch.empty(F, N, dtype=vt, device="cuda")
    else:
        st["Q"] = _random((len(_emitter_vertices(p)),), seed, torch.float32)
        st["out"] = torch.empty(F, N, dtype=torch.float32, device="cuda")
    return st


def _temperature(case, T):
    # FP32 operators: the temperatures follow from FP32 intensities, and a consumer stores them as such
    return T if _vector_type(case) == torch.float64 else T.float()


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "apply":
        state["op"].apply(state["X"], state["Y"])
        return state["Y"]
    if kind == "solve":
        op = rt.rt_build_operator(state["problem"], state["hp"])
        op.solve_fixed_point(state["J"], state["T"], tol=case["tol"], max_iter=300, check_every=4,
                             refine_tol=_refine_tol(case))
        op.free()
        return state["J"], _temperature(case, state["T"])
    if kind == "source":
        so = rt.rt_build_source_operator(state["op"])
        so.apply(state["Q"], state["out"])
        so.free()
        return state["out"]
    if kind == "batch":
        b = rt.rt_build_batch(state["problems"], state["hp"], threads=16, tune=False)
        info = b.info()
        J = torch.empty(info["total_vec"], dtype=torch.float32, device="cuda")
        T = torch.empty(info["total_vert"], dtype=torch.float64, device="cuda")
        b.solve(J, T, tol=case["tol"], max_iter=300, check_every=4)
        b.free()
        return J, T.float()
    srv = state["server"]
    ids = [srv.submit(p) for p in state["problems"]]
    out = []
    for rid in ids:
        J, T, _ = srv.poll(rid, wait_ms=60000)
        out.append((J, T.astype(np.float32)))
    return out


# ------------------------------------------------------------------- the work
def _entries(N, dense):
    """Stored entries of one operator: near blocks of 64-row leaves plus rank r (m + n) far blocks
    (the measured compression of the default parameters)."""
    if dense or N <= 1000:
        return float(N) * N
    return N * min(float(N), 937.0 * (math.log2(N) - 9.4))


def _assembly(N, G, dense, terms=2):
    """Kernel values needed for the stored entries, every point of a tetrahedron once per row, and their cost."""
    values = _entries(N, dense) * 24.0 * terms
    return values * (TERMS_FLOPS + 4.0 * G)


def _apply_bytes(N, F, G, dense, item, far):
    e = _entries(N, dense)
    near = e if dense else min(e, 1700.0 * N)
    return G * (near * item + (e - near) * far) + 2.0 * F * N * item


def _solve_work(N, F, G, dense, terms=2):
    tets = 6.0 * N
    return dict(bytes=24.0 * N + 16.0 * tets + 4.0 * F * N + 8.0 * N, flops=_assembly(N, G, dense, terms))


def work(case):
    if case["kind"] in ("batch", "serve"):
        each = [_solve_work(n ** 3, F, F, False) for n, F in _sizes(case)]
        return dict(bytes=sum(w["bytes"] for w in each), flops=sum(w["flops"] for w in each))
    dense = case["mode"] == "dense"
    F = 1 if case["grey"] else case["F"]
    G = 1 if case["shared"] or case["grey"] else (case["bins"] or F)
    if case["geometry"] == "box":
        n = case["n"]
        return _solve_work((3 * n // 5 + 1) ** 2 * (n + 1), F, G, False, terms=7)
    N = case["n"] ** 3
    if case["kind"] == "solve":
        return _solve_work(N, F, G, dense)
    if case["kind"] == "source":
        L, tri = case["n"] ** 2, 2 * (case["n"] - 1) ** 2
        return dict(bytes=4.0 * F * N + 4.0 * L, flops=N * tri * 3.0 * 2 * (TERMS_FLOPS + 3.0 * G))
    item = 8 if _vector_type(case) == torch.float64 else 4
    far = 2 if case["prec"] in ("bf16", "f16") else item
    reads = 1 if G == 1 and case["prec"] in ("bf16", "f16") else F / G
    b = _apply_bytes(N, F, G, dense, item, far)
    return dict(bytes=b * max(1.0, reads), flops=2.0 * F * _entries(N, dense))


# -------------------------------------------------- what 64-bit arithmetic gives
_A4, _B4 = (5.0 + 3.0 * math.sqrt(5.0)) / 20.0, (5.0 - math.sqrt(5.0)) / 20.0


def _tet_rules(dev):
    """Barycentric points and weights: the 4-point rule of degree 2, the 14-point rule of degree 5."""
    r4 = [([_A4 if d == k else _B4 for d in range(4)], 0.25) for k in range(4)]
    r14 = []
    for a, w in ((0.0927352503108912, 0.07349304311636196), (0.3108859192633006, 0.1126879257180159)):
        r14 += [([1.0 - 3.0 * a if d == k else a for d in range(4)], w) for k in range(4)]
    s = 0.4544962958743504
    r14 += [([s if d in (a, c) else 0.5 - s for d in range(4)], 0.04254602077708147)
            for a in range(4) for c in range(a + 1, 4)]
    f = lambda v: torch.tensor(v, dtype=torch.float64, device=dev)  # noqa: E731
    return [(f([b for b, _ in r]), f([w for _, w in r])) for r in (r4, r14)]


def _tri_rules(dev):
    r3 = [([2 / 3 if d == k else 1 / 6 for d in range(3)], 1 / 3) for k in range(3)]
    q = math.sqrt(15.0)
    r7 = [([1 / 3] * 3, 0.225)]
    for a, w in (((6 - q) / 21, (155 - q) / 1200), ((6 + q) / 21, (155 + q) / 1200)):
        r7 += [([1 - 2 * a if d == k else a for d in range(3)], w) for k in range(3)]
    f = lambda v: torch.tensor(v, dtype=torch.float64, device=dev)  # noqa: E731
    return [(f([b for b, _ in r]), f([w for _, w in r])) for r in (r3, r7)]


class _Exact:
    """The dense operator and source of one cube problem (at most one wall, z = 0) in 64 bits."""

    def __init__(self, p, bins=0):
        self.dev = "cuda" if torch.cuda.is_available() else "cpu"
        t = lambda a: torch.tensor(np.asarray(a), device=self.dev)  # noqa: E731
        self.p, self.x, self.tet, self.tri = p, t(p.xyz), t(p.tet).long(), t(p.emit_tri).long()
        self.nu, self.w, self.c, self.a = (t(v)[:, None] for v in (p.freqs.nu, p.freqs.w, p.freqs.c, p.freqs.albedo))
        self.k0, self.amp, self.R0 = p.kappa.k0, p.kappa.amp, p.wall.R0
        self.scales, self.group = torch.unique(self.c[:, 0], return_inverse=True)
        self.flip = torch.tensor([1.0, 1.0, -1.0], dtype=torch.float64, device=self.dev)

    def kappa(self, y):
        return self.k0 + self.amp * torch.sin(2 * math.pi * y).prod(-1)

    def depth(self, a, b):
        """int of kappa over the segment [a, b]: sin sin sin as four sinusoids, each integrated."""
        d = b - a
        L = d.norm(dim=-1)
        if self.amp == 0.0:
            return self.k0 * L
        m = a + 0.5 * d
        s = 0.0
        for sx, sy, sz, sign in ((1, 1, -1, 1), (-1, 1, 1, 1), (1, -1, 1, 1), (1, 1, 1, -1)):
            u = sx * m[..., 0] + sy * m[..., 1] + sz * m[..., 2]
            v = sx * d[..., 0] + sy * d[..., 1] + sz * d[..., 2]
            s = s + sign * torch.sin(2 * math.pi * u) * torch.sinc(v)
        return L * (self.k0 + 0.25 * self.amp * s)

    def path(self, x, y, reflected):
        """(source point, optical depth) of the direct or the reflected path from x to y."""
        if not reflected:
            return x, self.depth(x, y)
        src = x * self.flip
        den = y[..., 2:] - src[..., 2:]
        hit = src + torch.where(den > 0, -src[..., 2:] / den, torch.zeros_like(den)) * (y - src)
        return src, self.depth(x, hit) + self.depth(hit, y)

    def terms(self):
        return [(False, 1.0)] + ([(True, self.R0)] if self.R0 > 0 else [])

    def matrix(self):
        """G [groups, N, N]."""
        x, tet = self.x, self.tet
        N, T, C = x.shape[0], tet.shape[0], len(self.scales)
        V = x[tet]
        e = V[:, 1:] - V[:, :1]
        vol = torch.linalg.det(e).abs() / 6.0
        cen = V.mean(dim=1)
        lim = 4.0 * torch.stack([(V[:, i] - V[:, j]).square().sum(-1) for i in range(4) for j in range(i)]).amax(0)
        G = torch.zeros(C, N, N, dtype=torch.float64, device=self.dev)
        rules = _tet_rules(self.dev)
        pts = [torch.einsum("qk,tkd->tqd", b, V) for b, _ in rules]
        wts = [vol[:, None] * w * self.kappa(y) / (4 * math.pi) for y, (_, w) in zip(pts, rules)]
        rows = max(1, (1 << 23) // (4 * T))
        for r0 in range(0, N, rows):
            xi = x[r0:r0 + rows]
            R = xi.shape[0]
            for reflected, scale in self.terms():
                src = xi * self.flip if reflected else xi
                near = (src[:, None] - cen).square().sum(-1) < lim
                s, tau = self.path(xi[:, None, None], pts[0], reflected)
                geo = scale * wts[0] / (s - pts[0]).square().sum(-1) * (~near)[:, :, None]
                ri, ti = near.nonzero(as_tuple=True)
                sn, taun = self.path(xi[ri][:, None], pts[1][ti], reflected)
                geon = scale * wts[1][ti] / (sn - pts[1][ti]).square().sum(-1)
                for g in range(C):
                    cg = float(self.scales[g])
                    v = (cg * geo * torch.exp(-cg * tau)) @ rules[0][0]
                    vn = (cg * geon * torch.exp(-cg * taun)) @ rules[1][0]
                    v = v.index_put((ri, ti), vn, accumulate=True)
                    G[g, r0:r0 + R].index_add_(1, tet.reshape(-1), v.reshape(R, -1))
        return G

    def emitted(self, Q):
        """The source [F, N] for emitter coefficients Q [N] (read at the emitter's vertices)."""
        x = self.x
        out = torch.zeros(len(self.scales), x.shape[0], dtype=torch.float64, device=self.dev)
        V = x[self.tri]
        n = torch.linalg.cross(V[:, 1] - V[:, 0], V[:, 2] - V[:, 0])
        area2 = n.norm(dim=-1)
        n = n / area2[:, None]
        cen = V.mean(dim=1)
        lim = 4.0 * torch.stack([(V[:, i] - V[:, j]).square().sum(-1) for i in range(3) for j in range(i)]).amax(0)
        rules = _tri_rules(self.dev)
        rows = max(1, (1 << 22) // (7 * self.tri.shape[0]))
        angle = []
        for k in range(3):
            u, v = V[:, (k + 1) % 3] - V[:, k], V[:, (k + 2) % 3] - V[:, k]
            angle.append(torch.acos(((u * v).sum(-1) / (u.norm(dim=-1) * v.norm(dim=-1))).clamp(-1, 1)))
        for r0 in range(0, x.shape[0], rows):
            xi = x[r0:r0 + rows]
            ids = torch.arange(r0, r0 + xi.shape[0], device=self.dev)
            for reflected, scale in self.terms():
                src = xi * self.flip if reflected else xi
                at_x = (src - xi).square().sum(-1) <= 1e-20
                own = (self.tri[None] == ids[:, None, None]) & at_x[:, None, None]
                cm = -((src[:, None] - V[:, 0]) * n).sum(-1)
                near = (src[:, None] - cen).square().sum(-1) < lim
                for (b, w), use in zip(rules, (~near, near)):
                    y = torch.einsum("qk,tkd->tqd", b, V)
                    q = Q[self.tri] @ b.T
                    s, tau = self.path(xi[:, None, None], y, reflected)
                    keep = use & (cm > 0) & ~own.any(-1)
                    r2 = (s - y).square().sum(-1)
                    geo = torch.where(keep[:, :, None], scale * 0.5 * area2[:, None] * w * q * cm[:, :, None] ** 2 /
                                      (r2 * r2) / (4 * math.pi), torch.zeros_like(r2))
                    for g in range(len(self.scales)):
                        out[g, r0:r0 + rows] += (geo * torch.exp(-self.scales[g] * tau)).sum((1, 2))
                lim_term = sum((own[:, :, k] * angle[k]).sum(1) for k in range(3)) * scale / (8 * math.pi) * Q[ids]
                out[:, r0:r0 + rows] += lim_term
        full = out[self.group]
        return full * (SIGMA * self.p.T_emit ** 4 if self.p.grey else self.planck(self.p.T_emit))

    def planck(self, T):
        T = torch.as_tensor(T, dtype=torch.float64, device=self.dev)
        x = self.nu / T.clamp_min(1e-300)
        return torch.where((T > 0) & (x < 700), self.nu ** 3 / torch.expm1(x.clamp_max(700.0)), torch.zeros_like(x))

    def temperature(self, J):
        if self.p.grey:
            return (J[0].clamp_min(0) / SIGMA) ** 0.25
        wt = self.w * self.c * (1 - self.a)
        rhs = (wt * J).sum(0)
        lo, hi = torch.zeros_like(rhs), torch.ones_like(rhs)
        while bool(((wt * self.planck(hi)).sum(0) < rhs).any()):
            hi = 2 * hi
        for _ in range(70):
            mid = 0.5 * (lo + hi)
            low = (wt * self.planck(mid)).sum(0) < rhs
            lo, hi = torch.where(low, mid, lo), torch.where(low, hi, mid)
        return 0.5 * (lo + hi)

    def apply(self, G, X):
        return torch.stack([G[int(g)] @ X[f] for f, g in enumerate(self.group)])

    def solve(self, tol, every):
        G, E = self.matrix(), self.emitted(torch.full((self.x.shape[0],), self.p.Q0, dtype=torch.float64, device=self.dev))
        J, T = torch.zeros_like(E), torch.zeros_like(E[0])
        done = False
        while not done:
            for _ in range(every):
                B = SIGMA * T[None] ** 4 if self.p.grey else self.planck(T)
                new = E + self.apply(G, self.a * J + (1 - self.a) * B)
                done = done or bool((new - J).norm() <= tol * new.norm())
                J = new
                T = self.temperature(J)
        return J, T


def exact(case, seed):
    if case["geometry"] != "cube" or case["kind"] in ("batch", "serve") or case["bins"]:
        return None
    F = 1 if case["grey"] else case["F"]
    N, G = case["n"] ** 3, 1 if case["shared"] or case["grey"] else F
    if case["kind"] == "source":
        p = _one(case, seed)
        ids = _emitter_vertices(p)
        Q = torch.zeros(N, dtype=torch.float64, device="cuda")
        Q[torch.tensor(ids, device="cuda").long()] = _random((len(ids),), seed, torch.float32).double()
        return _Exact(p).emitted(Q)
    if N > 7000 or float(N) * N * (10 + G) > 1e9:
        return None
    ex = _Exact(_one(case, seed))
    if case["kind"] == "apply":
        return ex.apply(ex.matrix(), _random((F, N), seed, _vector_type(case)).double())
    return ex.solve(case["tol"], 4)
