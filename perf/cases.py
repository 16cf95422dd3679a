"""Performance cases of the scabem operator: the calls that users of the library make, over the
sizes they make them at, with inputs made from a seed and a plain FP64 reference of each result.

A case names a mesh (a straight guide, a directional coupler or a sphere), a grid, the precision and
the call (``path``):

* ``apply`` / ``adjoint``  y = A x or x = A^T y, the call inside every Krylov iteration;
* ``solve``     right-hand sides and GMRES with FP64 refinement, the call of one excitation or of a
                batch of excitations;
* ``gradient``  one step of an absorber-profile optimisation: the differentiable solve forward and
                backward through the adjoint system;
* ``post``      reflection fit on the guide's axis and E, H on a cross-section, after a solve;
* ``sweep``     one point of a wavelength sweep: a new operator, its conductivity and right-hand
                side, and one product with it.

``prepare`` builds what a program has in hand before the call (the operator, vectors, sources) and
``run`` makes the call.  ``exact`` evaluates the same grid operator in FP64 with torch alone.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_1004_5076_gb300 as sc
from paper_1004_5076_gb300.autograd import absorber_solve

ETA0 = 376.730313668
DEV = "cuda" if torch.cuda.is_available() else "cpu"


# ------------------------------------------------------------------ cases
def _guide(name, path, length, nx, ny, nz, absorber, px, py, pz, near_h=2.05, prec=64, nrhs=1, lam=1.55, p=3, q=6):
    return {"name": name, "path": path, "mesh": "guide", "length": length, "nx": nx, "ny": ny, "nz": nz,
            "absorber": absorber, "px": px, "py": py, "pz": pz, "p": p, "q": q, "near_h": near_h, "prec": prec,
            "nrhs": nrhs, "lam": lam}


def _sphere(name, path, level, n, near_h, prec=64, nrhs=1, lam=1.55):
    return {"name": name, "path": path, "mesh": "sphere", "level": level, "px": n, "py": n, "pz": n, "p": 3, "q": 6,
            "near_h": near_h, "prec": prec, "nrhs": nrhs, "lam": lam}


def listed():
    g12 = dict(length=12.0, nx=300, ny=11, nz=5, absorber=4.0, px=512, py=64, pz=64)
    return [
        # the dielectric sphere of 320 triangles: the smallest operator in use, where launches count
        _sphere("apply-sphere-320", "apply", 2, 32, 4.0),
        # the 12 um guide, the operator of the paper's experiments: one Krylov vector ...
        _guide("apply-guide-12um", "apply", **g12),
        # ... the eight columns of a lockstep solve ...
        _guide("apply-guide-12um-x8", "apply", nrhs=8, **g12),
        # ... the FP64 product of the refinement residual and of complex128 solves ...
        _guide("apply-guide-12um-c128", "apply", prec=128, **g12),
        # ... and the transposed product of adjoint solves
        _guide("adjoint-guide-12um", "adjoint", **g12),
        # a closed body whose active columns fill the cross-section (FFT planes), the more accurate
        # near radius and an odd number of columns
        _sphere("apply-sphere-5120-x3", "apply", 4, 64, 3.05, nrhs=3),
        # the directional coupler: the largest operator in use
        {"name": "apply-coupler-40um", "path": "apply", "mesh": "coupler", "length": 40.0, "nx": 1000, "ny": 11,
         "nz": 5, "absorber": 4.0, "px": 1024, "py": 256, "pz": 256, "p": 3, "q": 6, "near_h": 2.05, "prec": 64,
         "nrhs": 1, "lam": 1.55},
        # one excitation solved on a short guide, and eight in lockstep on a longer one
        _guide("solve-guide-2um", "solve", 2.0, 40, 6, 3, 0.6, 64, 32, 16, near_h=3.05),
        _guide("solve-guide-3um-x8", "solve", 3.0, 60, 4, 2, 0.75, 64, 16, 16, near_h=2.05, nrhs=8),
        # one step of an absorber optimisation with 16 B-spline coefficients
        _guide("gradient-guide-1.6um", "gradient", 1.6, 16, 4, 2, 0.4, 32, 16, 16, near_h=3.05),
        # reflection and fields after a solve of the 12 um guide
        _guide("post-guide-12um", "post", **g12),
        # one wavelength of a sweep on a mid-size guide with an odd mesh
        _guide("sweep-guide-5um", "sweep", 5.0, 123, 9, 5, 1.3, 256, 32, 16, lam=1.31),
    ]


def _unnamed(c):
    return {k: v for k, v in c.items() if k != "name"}


def draw(rng):
    """One more case of the same ranges."""
    path = rng.choice(["apply", "apply", "apply", "apply", "adjoint", "adjoint", "solve", "gradient", "post", "sweep"])
    prec = rng.choice([64, 64, 64, 128]) if path in ("apply", "adjoint", "sweep") else 64
    near_h = rng.choice([2.05, 2.05, 3.05])
    lam = rng.uniform(1.25, 1.65)
    nrhs = rng.choice([1, 1, 1, 2, 3, 5, 8]) if path in ("apply", "solve") else rng.choice([1, 2]) if path == "adjoint" else 1
    if path in ("apply", "adjoint") and rng.random() < 0.25:
        level, n = rng.choice([(2, 32), (3, 32), (4, 32), (3, 64), (4, 64)])
        return _unnamed(_sphere("", path, level, n, rng.choice([2.05, 3.05, 4.0]), prec, nrhs, lam))
    lo, hi = {"solve": (1.2, 2.4), "gradient": (1.2, 2.0), "sweep": (1.5, 6.0)}.get(path, (1.0, 16.0))
    length = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    fine = path not in ("solve", "gradient")
    nx = max(8, round(length * rng.uniform(*((12, 26) if fine else (10, 16)))))
    ny, nz = (rng.randint(4, 11), rng.randint(2, 5)) if fine else (rng.randint(3, 5), rng.randint(2, 3))
    absorber = length * rng.uniform(0.15, 0.35)
    # the smallest transforms whose spacing is at most the mesh spacing along the guide and 0.08 um
    h, p = min(0.08, 1.15 * length / nx), rng.choice([3, 3, 3, 3, 2, 4])
    px, py, pz = ((8 if s == 0 else 4) for s in range(3))
    for _ in range(12):
        px = px * 2 if length / (px // 2 - p - 1.5) > h or px // 2 - p < 2 else px
        py = py * 2 if py // 2 - p < 2 or 0.5 / (py // 2 - p - 1.5) > h else py
        pz = pz * 2 if pz // 2 - p < 2 or 0.22 / (pz // 2 - p - 1.5) > h else pz
    return _unnamed(_guide("", path, length, nx, ny, nz, absorber, min(px, 1024), py, pz, near_h, prec, nrhs, lam, p))


# ------------------------------------------------------------------ meshes, grids, profiles
def _box(x, y, z):
    """Structured closed surface of a box from its node coordinates, oriented outward."""
    nx, ny, nz = len(x) - 1, len(y) - 1, len(z) - 1
    i, j, k = np.meshgrid(np.arange(nx + 1), np.arange(ny + 1), np.arange(nz + 1), indexing="ij")
    node = (i * (ny + 1) + j) * (nz + 1) + k
    faces = []
    for ids in (node[0].T, node[nx], node[:, 0], node[:, ny].T, node[:, :, 0].T, node[:, :, nz]):
        a, b, c, d = ids[:-1, :-1], ids[1:, :-1], ids[1:, 1:], ids[:-1, 1:]
        faces.append(np.stack([np.stack([a, b, c], -1), np.stack([a, c, d], -1)], -2).reshape(-1, 3))
    T = np.concatenate(faces)
    used, T = np.unique(T, return_inverse=True)
    xyz = np.stack([np.asarray(x)[i.ravel()], np.asarray(y)[j.ravel()], np.asarray(z)[k.ravel()]], -1)
    return xyz[used], T.reshape(-1, 3).astype(np.int32)


def _icosphere(level):
    t = (1 + math.sqrt(5)) / 2
    V = np.array([(-1, t, 0), (1, t, 0), (-1, -t, 0), (1, -t, 0), (0, -1, t), (0, 1, t), (0, -1, -t), (0, 1, -t),
                  (t, 0, -1), (t, 0, 1), (-t, 0, -1), (-t, 0, 1)], dtype=float)
    D = np.linalg.norm(V[:, None] - V[None], axis=-1)
    near = (D > 0) & (D < 2.1)
    T = np.array([(a, b, c) for a in range(12) for b in range(a) for c in range(b) if near[a, b] and near[b, c] and near[a, c]])
    V /= np.linalg.norm(V, axis=1, keepdims=True)
    for _ in range(level):
        e = np.sort(np.stack([T[:, [0, 1]], T[:, [1, 2]], T[:, [2, 0]]], 1).reshape(-1, 2), axis=1)
        u, inv = np.unique(e, axis=0, return_inverse=True)
        m = inv.reshape(-1, 3) + len(V)
        mid = V[u[:, 0]] + V[u[:, 1]]
        V = np.concatenate([V, mid / np.linalg.norm(mid, axis=1, keepdims=True)])
        a, b, c = T.T
        ab, bc, ca = m.T
        T = np.concatenate([np.stack(s, 1) for s in ((a, ab, ca), (b, bc, ab), (c, ca, bc), (ab, bc, ca))])
    flip = np.einsum("ij,ij->i", np.cross(V[T[:, 1]] - V[T[:, 0]], V[T[:, 2]] - V[T[:, 0]]), V[T].mean(1)) < 0
    T[flip] = T[flip][:, [0, 2, 1]]
    return V, T.astype(np.int32)


def _mesh(c):
    """Vertices, triangles and absorber flags of a case."""
    if c["mesh"] == "sphere":
        V, T = _icosphere(c["level"])
        return V, T, (V[T].mean(1)[:, 0] > 0.2).astype(np.int32)
    x = np.linspace(0.0, c["length"], c["nx"] + 1)
    y, z = np.linspace(-0.25, 0.25, c["ny"] + 1), np.linspace(-0.11, 0.11, c["nz"] + 1)
    V, T = _box(x, y, z)
    if c["mesh"] == "coupler":  # two guides 0.2 um apart
        T = np.concatenate([T, T + len(V)])
        V = np.concatenate([V - [0, 0.35, 0], V + [0, 0.35, 0]])
    cx = V[T].mean(1)[:, 0]
    return V, T.astype(np.int32), ((cx < c["absorber"]) | (cx > c["length"] - c["absorber"])).astype(np.int32)


def _media(c):
    return (2.25, 1.0, 1.0, 1.0, c["lam"]) if c["mesh"] == "sphere" else (12.1, 1.0, 2.1, 1.0, c["lam"])


def _grid(c, V):
    """Physical points per axis, spacing and origin of the uniform grid around V."""
    n, p = (c["px"] // 2, c["py"] // 2, c["pz"] // 2), c["p"]
    lo, hi = V.min(0), V.max(0)
    h = float(max((hi - lo)[a] / (n[a] - p - 1.5) for a in range(3)))
    off = (0.236, 0.382, 0.146)  # keeps the points of structured meshes off cell boundaries
    return n, h, tuple(float((lo + hi)[a] / 2 - h * ((n[a] - 1) / 2 - off[a])) for a in range(3))


def _sigma(c, seed, nt, region):
    """Arguments of scabem_set_sigma: graded absorbers at both ends of a guide, a random sheet on a sphere."""
    rng = np.random.default_rng(seed)
    if c["mesh"] == "sphere":
        return {"per_qpoint": rng.uniform(0.0, 3e-3, (nt, c["q"])) * region[:, None]}
    if c["path"] == "gradient":
        return {"bspline": (0.0, c["length"], 0, rng.uniform(1e-3, 8e-3, 16))}
    L, s0 = c["absorber"], rng.uniform(4e-3, 1.2e-2)
    return {"segments": [(c["length"] - L, L, s0, 3, 0, 1.0), (L, L, s0, 3, 0, -1.0)]}


def _sources(c, seed):
    """Beams and dipoles in the plain section of a guide, one per right-hand side (argument dicts)."""
    rng = np.random.default_rng([seed, 1])
    a, b = c["absorber"] + 0.1 * c["length"], 0.6 * c["length"] - 0.2 * c["absorber"]
    out = []
    for i in range(c["nrhs"]):
        pos = (float(rng.uniform(a, b)), float(rng.uniform(-0.03, 0.03)), float(rng.uniform(-0.02, 0.02)))
        pol = (0.0, 1.0, 0.0) if i % 2 == 0 else (0.0, 0.0, 1.0)
        out.append(dict(kind="beam", pos=pos, dir=(1.0, 0.0, 0.0), pol=pol, b=0.07))
    return out


def _receiver(c, seed):
    """A beam back along the guide: its tested field weighs the solution of an optimisation step."""
    rng = np.random.default_rng([seed, 3])
    return dict(kind="beam", pos=(float(rng.uniform(0.55, 0.62) * c["length"]), 0.01, 0.0), dir=(-1.0, 0.0, 0.0),
                pol=(0.0, 1.0, 0.0), b=0.07)


def _vectors(seed, rows, n, dtype):
    rng = np.random.default_rng([seed, 2])
    v = (rng.standard_normal((rows, n)) + 1j * rng.standard_normal((rows, n))) / math.sqrt(2)
    return torch.as_tensor(v).to(dtype)


def _probe(c):
    """Probe line of the reflection fit and a cross-section of points inside the guide."""
    t0, t1 = 0.5 * c["length"], c["length"] - c["absorber"]
    y, z = np.meshgrid(np.linspace(-0.2, 0.2, 9), np.linspace(-0.08, 0.08, 7), indexing="ij")
    pts = np.stack([np.full(y.size, 0.45 * c["length"]), y.ravel(), z.ravel()], -1)
    return dict(p0=(0.0, 0.01, -0.005), t0=t0, t1=t1, npts=48, beta_lo=10.0, beta_hi=16.0, nbeta=601), pts


SOLVE = dict(tol=1e-5, restart=120, maxit=20000, refine_tol=1e-12, max_refine=20)


# ------------------------------------------------------------------ prepare / run
class _State:
    """What a program keeps: the mesh, the operator and its vectors.  Handles end with the state."""

    def __init__(self):
        self.op = self.mesh = None

    def __del__(self):
        if self.op is not None:
            sc.scabem_op_destroy(self.op)
        if self.mesh is not None:
            sc.scabem_mesh_destroy(self.mesh)


def _create(c, mesh, V):
    n, h, origin = _grid(c, V)
    mask = 3 if c["mesh"] != "coupler" else 1 if c["prec"] == 64 else 2  # the coupler in the one precision it runs in
    return sc.scabem_op_create(mesh, _media(c), n, h, origin, c["p"], c["q"], c["near_h"] * h, mask)


def prepare(case, seed):
    c, s = case, _State()
    V, T, region = _mesh(c)
    s.case, s.V = c, V
    s.mesh = sc.scabem_mesh_create(V, T, region)
    s.N = sc.scabem_mesh_info(s.mesh)[2]
    s.prec, s.dtype = (sc.SCABEM_C64, torch.complex64) if c["prec"] == 64 else (sc.SCABEM_C128, torch.complex128)
    s.sigma = _sigma(c, seed, len(T), region)
    if c["path"] != "sweep":
        s.op = _create(c, s.mesh, V)
        if c["path"] != "gradient":
            sc.scabem_set_sigma(s.op, **s.sigma)
    if c["mesh"] != "sphere":
        s.sources = [sc.make_source(side="i", **k) for k in _sources(c, seed)]
    if c["path"] in ("apply", "adjoint", "sweep"):
        s.x = _vectors(seed, c["nrhs"], s.N, s.dtype).to(DEV)
        s.y = torch.empty_like(s.x)
    elif c["path"] == "post":
        s.x = _vectors(seed, 1, s.N, torch.complex128).to(DEV)
    elif c["path"] == "gradient":
        s.coef = torch.tensor(s.sigma["bspline"][3], requires_grad=True)
        s.receiver = torch.empty(s.N, dtype=torch.complex128, device=DEV)
        sc.scabem_rhs(s.op, [sc.make_source(side="i", **_receiver(c, seed))], s.receiver)
    return s


def run(state):
    s, c = state, state.case
    if c["path"] in ("apply", "adjoint"):
        call = sc.scabem_apply if c["path"] == "apply" else sc.scabem_apply_adjoint
        call(s.op, s.x, s.y, nrhs=c["nrhs"], ld=s.N, prec=s.prec)
        return s.y
    if c["path"] == "solve":
        b = torch.empty((c["nrhs"], s.N), dtype=torch.complex128, device=DEV)
        sc.scabem_rhs(s.op, s.sources, b, ld=s.N)
        x = torch.zeros_like(b)
        sc.scabem_solve(s.op, b, x, nrhs=c["nrhs"], ld=s.N, prec=sc.SCABEM_C64, **SOLVE)
        return x
    if c["path"] == "gradient":
        s.coef.grad = None
        x = absorber_solve(s.coef, s.op, s.N, s.sigma["bspline"][:3], s.sources, prec=sc.SCABEM_C64, **SOLVE)
        torch.dot(s.receiver, x).abs().square().backward()  # the power a second beam receives
        return [x.detach(), s.coef.grad]
    if c["path"] == "post":
        probe, pts = _probe(c)
        r = sc.scabem_reflection(s.op, s.x, 0, 1, inc=s.sources[0], ld=s.N, **probe)
        E, H = sc.scabem_fields_eh(s.op, s.x, pts, side=0, inc=s.sources[0], ld=s.N)
        return [r, E, H]
    op = _create(c, s.mesh, s.V)
    try:
        sc.scabem_set_sigma(op, **s.sigma)
        b = torch.empty_like(s.x)
        sc.scabem_rhs(op, s.sources, b, ld=s.N, prec=s.prec)
        sc.scabem_apply(op, s.x, s.y, nrhs=1, ld=s.N, prec=s.prec)
        torch.cuda.synchronize()
    finally:
        sc.scabem_op_destroy(op)
    return [b, s.y]


# ------------------------------------------------------------------ work
def work(case):
    """Bytes and operations of one pass that no implementation of the path avoids: every vector and
    every conductivity in and out once, one pass over the near interactions between edges (three
    values per pair of plain edges, eight per pair of absorber edges), the products with them and the
    transforms of 12 and 16 fields on the active box."""
    c = case
    if c["mesh"] == "sphere":
        nt, absorbing, size, area = 20 * 4 ** c["level"], 0.4, (2.0, 2.0, 2.0), 12.6
    else:
        k = 2 if c["mesh"] == "coupler" else 1
        nt = k * 4 * (c["nx"] * (c["ny"] + c["nz"]) + c["ny"] * c["nz"])
        absorbing, size = 2 * c["absorber"] / c["length"], (c["length"], 0.5 if k == 1 else 1.2, 0.22)
        area = k * 1.44 * c["length"]
    n = (c["px"] // 2, c["py"] // 2, c["pz"] // 2)
    h = max(size[a] / (n[a] - c["p"] - 1.5) for a in range(3))
    near = nt * min(nt, math.pi * (c["near_h"] * h) ** 2 * nt / area)
    N = 1.5 * nt * (2 + absorbing)
    word, k = c["prec"] // 8, c["nrhs"]
    entries = 2.25 * near * (3 + 5 * absorbing)
    box = math.prod(min(2 * n[a], size[a] / h + c["p"]) for a in range(3))
    flops = k * (8 * entries + 28 * 5 * box * math.log2(max(box, 2)))
    moved = word * (2 * k * N + entries) + 8 * nt * c["q"]
    if c["path"] == "post":  # 48 + 63 points against every source point: 9 and 18 complex sums
        points = 48 * 9 + 63 * 18
        return {"bytes": 16 * N + 48 * points, "flops": 8.0 * points * nt * c["q"] + 601 * 48 * 40}
    if c["path"] in ("solve", "gradient"):  # about 700 iterations per solve
        its = 700 * (2 if c["path"] == "gradient" else 1)
        return {"bytes": its * (moved + 16 * N * k), "flops": its * (flops + 16 * N * k)}
    if c["path"] == "sweep":  # the panel integrals of every near pair at every point, both media
        flops += near * c["q"] * 2 * (c["q"] * 60 + 300)
    return {"bytes": moved, "flops": flops}


# ------------------------------------------------------------------ exact (FP64, torch only)
def _lagrange(t, p):
    L, D = [], []
    for i in range(p):
        v, d = torch.ones_like(t), torch.zeros_like(t)
        for m in range(p):
            if m != i:
                v = v * (t - m) / (i - m)
                term = torch.ones_like(t) / (i - m)
                for r in range(p):
                    if r not in (i, m):
                        term = term * (t - r) / (i - r)
                d = d + term
        L.append(v)
        D.append(d)
    return torch.stack(L, -1), torch.stack(D, -1)


class _Reference:
    """The grid-accelerated PMCHW operator with absorber rows, stage by stage in FP64."""

    def __init__(self, c):
        V, T, region = _mesh(c)
        self.c, self.p, self.q = c, c["p"], c["q"]
        ei, mi, ee, me, lam = _media(c)
        w = 2 * math.pi / lam
        self.k, self.z = (w * math.sqrt(ee * me), w * math.sqrt(ei * mi)), (math.sqrt(me / ee), math.sqrt(mi / ei))
        self.n, self.h, self.origin = _grid(c, V)
        self.region = region
        self._edges(T, region)
        t64 = dict(dtype=torch.float64, device=DEV)
        tv = torch.as_tensor(V[T], **t64)
        self.nt = len(T)
        cr = torch.linalg.cross(tv[:, 1] - tv[:, 0], tv[:, 2] - tv[:, 0])
        area = cr.norm(dim=1) / 2
        self.tv, self.normal, self.cen = tv, cr / cr.norm(dim=1, keepdim=True), tv.mean(1)
        a, b = 0.445948490915965, 0.091576213509771  # the six-point rule
        bary = torch.tensor([[a + (1 - 3 * a) * (i == j) for j in range(3)] for i in range(3)]
                            + [[b + (1 - 3 * b) * (i == j) for j in range(3)] for i in range(3)], **t64)
        wq = torch.tensor([0.223381589678011] * 3 + [0.109951743655322] * 3, **t64)
        self.r = torch.einsum("aj,tjc->tac", bary, tv)
        self.w = wq * area[:, None]
        self.rel, self.relv = self.r - self.cen[:, None], tv - self.cen[:, None]
        length = torch.stack([(tv[:, (k + 2) % 3] - tv[:, (k + 1) % 3]).norm(dim=1) for k in range(3)], 1)
        self.cX = torch.as_tensor(self.sign, **t64) * length / (2 * area[:, None])
        self.X = self.cX[:, :, None, None] * (self.r[:, None] - tv[:, :, None])  # (nt, k, q, 3)
        self.nX = torch.linalg.cross(self.normal[:, None, None].expand_as(self.X), self.X)
        self._stencils()
        self.G = [self._green(k) for k in self.k]
        self.near = None

    def _edges(self, T, region):
        e = np.stack([T[:, [1, 2]], T[:, [2, 0]], T[:, [0, 1]]], 1).astype(np.int64)  # edge k is opposite vertex k
        self.sign = np.where(e[..., 0] < e[..., 1], 1, -1)
        key = e.min(-1) * (T.max() + 1) + e.max(-1)
        u, inv = np.unique(key, return_inverse=True)
        inv = inv.reshape(-1, 3)
        both = np.zeros(len(u))
        np.add.at(both, inv.ravel(), np.repeat(region, 3))
        plain = both < 2
        idx = np.where(plain, np.cumsum(plain) - 1, np.cumsum(~plain) - 1)
        nL, nR = int(plain.sum()), int((~plain).sum())
        self.N, self.nL, self.nR = 2 * nL + 3 * nR, nL, nR
        pl, ci = plain[inv], idx[inv]
        unk = np.stack([np.where(pl, ci, 2 * nL + ci), np.where(pl, ci, 2 * nL + nR + ci),
                        np.where(pl, nL + ci, 2 * nL + 2 * nR + ci)], -1)  # (nt, k, J_e J_i M)
        self.unk = torch.as_tensor(unk, device=DEV)
        self.usign = torch.as_tensor(np.stack([np.ones(pl.shape), np.where(pl, -1.0, 1.0), np.ones(pl.shape)], -1), device=DEV)
        row = np.full(pl.shape + (4,), self.N)  # index N collects the values without a row
        row[..., 0] = np.where(pl, ci, 2 * nL + ci)
        row[..., 1] = np.where(pl, nL + ci, self.N)
        row[..., 2] = np.where(pl, self.N, 2 * nL + nR + ci)
        row[..., 3] = np.where(pl, self.N, 2 * nL + 2 * nR + ci)
        self.row = torch.as_tensor(row, device=DEV)

    def _stencils(self):
        p, n = self.p, self.n
        u = (self.r.reshape(-1, 3) - torch.tensor(self.origin, dtype=torch.float64, device=DEV)) / self.h
        self.base = torch.floor(u - 0.5 * (p - 2)).long()
        self.L, D = _lagrange(u - self.base, p)
        self.D = D / self.h
        o = torch.arange(p, device=DEV)
        i, j, k = (v.reshape(-1) for v in torch.meshgrid(o, o, o, indexing="ij"))
        b = self.base
        self.gidx = ((b[:, 0:1] + i) * n[1] + b[:, 1:2] + j) * n[2] + b[:, 2:3] + k
        L, D = self.L, self.D
        self.W = L[:, 0, i] * L[:, 1, j] * L[:, 2, k]
        self.dW = torch.stack([D[:, 0, i] * L[:, 1, j] * L[:, 2, k], L[:, 0, i] * D[:, 1, j] * L[:, 2, k],
                               L[:, 0, i] * L[:, 1, j] * D[:, 2, k]], 1)

    def _green(self, k):
        d = []
        for n in self.n:
            i = torch.arange(2 * n, dtype=torch.float64, device=DEV)
            d.append(torch.where(i < n, i, i - 2 * n))
        R = self.h * (d[0][:, None, None] ** 2 + d[1][None, :, None] ** 2 + d[2][None, None, :] ** 2).sqrt()
        G = torch.polar(1 / (4 * math.pi * R), -k * R)
        G[0, 0, 0] = 0
        return G

    # ---- near corrections: exact panel moments minus the grid's own, per (pair, target point, medium)
    def _pairs(self):
        r2, out = (self.c["near_h"] * self.h) ** 2, []
        for t0 in range(0, self.nt, 2048):
            d2 = ((self.cen[t0:t0 + 2048, None] - self.cen[None]) ** 2).sum(-1)
            t, s = torch.nonzero(d2 < r2, as_tuple=True)
            out.append(torch.stack([t + t0, s]))
        return torch.cat(out, 1)

    def _static(self, r, s, same):
        """Closed-form integrals of 1/R, (rho' - rho)/R and grad(1/R) over source triangles s at r (m, q, 3)."""
        v, n = self.tv[s][:, None], self.normal[s][:, None].expand_as(r)
        d = torch.where(same[:, None], 0.0, ((r - v[:, :, 0]) * n).sum(-1))
        rho = r - d[..., None] * n
        I, om = torch.zeros_like(d), torch.zeros_like(d)
        Ir, gI = torch.zeros_like(r), torch.zeros_like(r)
        for e in range(3):
            a, b = v[:, :, e], v[:, :, (e + 1) % 3]
            l = (b - a) / (b - a).norm(dim=-1, keepdim=True)
            u = torch.linalg.cross(l.expand_as(n), n)
            sm, sp, t = ((a - rho) * l).sum(-1), ((b - rho) * l).sum(-1), ((a - rho) * u).sum(-1)
            r0 = t * t + d * d
            Rm, Rp = (r0 + sm * sm).sqrt(), (r0 + sp * sp).sqrt()
            f = torch.where(sp + sm > 0, torch.log((Rp + sp) / (Rm + sm)), torch.log((Rm - sm) / (Rp - sp)))
            be = torch.atan2(t * sp, r0 + d.abs() * Rp) - torch.atan2(t * sm, r0 + d.abs() * Rm)
            I, om = I + t * f - d.abs() * be, om + be
            Ir = Ir + 0.5 * u * (r0 * f + sp * Rp - sm * Rm)[..., None]
            gI = gI - u * f[..., None]
        return I, Ir, gI - n * (torch.sign(d) * om)[..., None], rho

    def _records(self, t, s, med):
        """(m, q, 10) corrections dP0, dP1, dQ, dC of the pairs (t, s)."""
        k, G, q, p = self.k[med], self.G[med], self.q, self.p
        r, c = self.r[t], self.cen[s][:, None]
        same = t == s
        I, Ir, gI, rho = self._static(r, s, same)
        D = r[:, :, None] - self.r[s][:, None]  # (m, a, b, 3)
        R = D.norm(dim=-1)
        own = same[:, None, None] & torch.eye(q, dtype=torch.bool, device=DEV)
        R = torch.where(own, 1.0, R)
        kr = k * R
        sh, sn, cn = torch.sin(kr / 2) ** 2, torch.sin(kr), torch.cos(kr)
        gv = torch.complex(-2 * sh / R, -sn / R)
        gd = torch.complex((2 * sh - kr * sn) / R ** 3, (sn - kr * cn) / R ** 3)
        gv, gd = torch.where(own, torch.tensor(-1j * k, dtype=gv.dtype, device=DEV), gv), torch.where(own, 0.0, gd)
        w, rel = self.w[s][:, None], self.rel[s][:, None]
        P0 = (I + (w * gv).sum(-1)) / (4 * math.pi)
        P1 = (Ir + (rho - c) * I[..., None] + ((w * gv)[..., None] * rel).sum(-2)) / (4 * math.pi)
        Q = (gI + ((w * gd)[..., None] * D).sum(-2)) / (4 * math.pi)
        C = torch.linalg.cross(Q, (r - c).to(Q.dtype))
        # the grid's interaction: weights per axis offset, then a (2p - 1)^3 window of the Green table
        at, bs = t[:, None] * q + torch.arange(q, device=DEV), s[:, None] * q + torch.arange(q, device=DEV)
        La, Da, Lb = self.L[at], self.D[at], self.L[bs]  # (m, q, axis, p)
        K = torch.zeros(t.shape[0], q, q, 3, 2 * p - 1, dtype=torch.float64, device=DEV)
        E = torch.zeros_like(K)
        for i in range(p):
            for j in range(p):
                K[..., i - j + p - 1] += La[:, :, None, :, i] * Lb[:, None, :, :, j]
                E[..., i - j + p - 1] += Da[:, :, None, :, i] * Lb[:, None, :, :, j]
        o = torch.arange(2 * p - 1, device=DEV) - (p - 1)
        dg = self.base[at][:, :, None] - self.base[bs][:, None]  # (m, a, b, 3)
        ix, iy, iz = (torch.remainder(dg[..., a, None] + o, 2 * self.n[a]) for a in range(3))
        win = G[ix[..., :, None, None], iy[..., None, :, None], iz[..., None, None, :]]  # (m, a, b, x, y, z)
        zc = torch.einsum("mabxyz,mabvz->vmabxy", win, torch.stack([K[..., 2, :], E[..., 2, :]], -2).to(win.dtype))
        Kx, Ky, Ex, Ey = (v.to(win.dtype) for v in (K[..., 0, :], K[..., 1, :], E[..., 0, :], E[..., 1, :]))
        y0, y1, y2 = ((v * u[..., None, :]).sum(-1) for v, u in ((zc[0], Ky), (zc[0], Ey), (zc[1], Ky)))
        gh = (y0 * Kx).sum(-1)
        gg = torch.stack([(y0 * Ex).sum(-1), (y1 * Kx).sum(-1), (y2 * Kx).sum(-1)], -1)
        P0 = P0 - (w * gh).sum(-1)
        P1 = P1 - ((w * gh)[..., None] * rel).sum(-2)
        Q = Q - (w[..., None] * gg).sum(-2)
        C = C - (w[..., None] * torch.linalg.cross(gg, rel.expand_as(gg).to(gg.dtype))).sum(-2)
        return torch.cat([P0[..., None], P1, Q, C], -1)

    def prepare_near(self):
        if self.near is None:
            pairs = self._pairs()
            step = max(1, int(3e8) // (16 * self.q ** 2 * (2 * self.p - 1) ** 3))
            self.near = [(pairs[0, i:i + step], pairs[1, i:i + step],
                          [self._records(pairs[0, i:i + step], pairs[1, i:i + step], m) for m in range(2)])
                         for i in range(0, pairs.shape[1], step)]

    # ---- the operator
    def currents(self, X):
        """Summaries (a, beta) of the J_e, J_i and M sets: (3, nt, B) and (3, nt, 3, B)."""
        j = self.cX[:, :, None, None] * (self.usign[..., None] * X[self.unk])  # (nt, k, set, B)
        return j.sum(1).permute(1, 0, 2), torch.einsum("tkc,tksb->stcb", self.relv.to(j.dtype), j)

    def _convolve(self, src, med):
        n, P = self.n, [2 * v for v in self.n]
        Gh = torch.fft.fftn(self.G[med]).unsqueeze(-1)
        out = []
        for f in src:  # (ng, B) each
            s = torch.fft.fftn(f.reshape(*n, -1), s=P, dim=(0, 1, 2))
            out.append(torch.fft.ifftn(Gh * s, dim=(0, 1, 2))[: n[0], : n[1], : n[2]].reshape(f.shape))
        return out

    def _interpolate(self, f, which):
        """Value (which = None) or derivative along an axis of grid field f at every point."""
        W = self.W if which is None else self.dW[:, which]
        out = 0
        for s in range(W.shape[1]):
            out = out + W[:, s, None] * f[self.gidx[:, s]]
        return out

    def fields(self, X):
        """Per medium the J and M potentials (A, phi, grad phi, curl) at the points."""
        nt, q, B = self.nt, self.q, X.shape[1]
        a, b = self.currents(X)
        self.a, self.b = a, b
        ng = math.prod(self.n)
        cols = []
        for s in range(3):
            J = self.w[..., None, None] * (self.rel[..., None] * a[s][:, None, None] - b[s][:, None])
            rho = (2 * self.w)[..., None] * a[s][:, None]
            cols.append([J[:, :, i].reshape(nt * q, B) for i in range(3)] + [rho.reshape(nt * q, B)])
        grids = []
        for s in range(3):
            gs = []
            for v in cols[s]:
                g = torch.zeros(ng, B, dtype=v.dtype, device=DEV)
                for e in range(self.W.shape[1]):
                    g = g.index_add(0, self.gidx[:, e], self.W[:, e, None] * v)
                gs.append(g)
            grids.append(gs)
        self.prepare_near()
        out = []
        for med in range(2):
            sets = []
            for s, sg in ((med, 1.0), (2, 1.0 if med == 0 else -1.0)):
                f = self._convolve(grids[s], med)
                A = [self._interpolate(f[i], None) for i in range(4)]
                g = [self._interpolate(f[3], i) for i in range(3)]
                d = lambda i, ax: self._interpolate(f[i], ax)  # noqa: E731
                cu = [d(2, 1) - d(1, 2), d(0, 2) - d(2, 0), d(1, 0) - d(0, 1)]
                F = torch.stack(A + g + cu, 1).reshape(nt, q, 10, B)
                for t, src, rec in self.near:
                    R = rec[med][..., None]
                    aS, bS = a[s][src][:, None], b[s][src][:, None]  # (m, 1, B), (m, 1, 3, B)
                    d0, d1, dq, dc = R[:, :, 0], R[:, :, 1:4], R[:, :, 4:7], R[:, :, 7:10]
                    add = torch.cat([d1 * aS[:, :, None] - d0[:, :, None] * bS, 2 * (d0 * aS)[:, :, None],
                                     2 * dq * aS[:, :, None],
                                     dc * aS[:, :, None] - torch.linalg.cross(dq.expand(*dq.shape[:3], B), bS.expand(-1, q, -1, -1), dim=2)], 2)
                    F = F.index_add(0, t, add)
                sets.append(sg * F)
            out.append(sets)
        return out

    def apply(self, X, sigma):
        """A X for X (N, B) and conductivities sigma (nt, q) in siemens."""
        F = self.fields(X)
        sg = (sigma * ETA0)[..., None, None]
        WE = WH = wE = wH = 0
        E = []
        for med, (J, M) in enumerate(F):
            k, z, sgn = self.k[med], self.z[med], 1.0 if med == 0 else -1.0
            A, phi, gphi, cA, Fm, psi, cF = J[:, :, :3], J[:, :, 3], J[:, :, 4:7], J[:, :, 7:], M[:, :, :3], M[:, :, 3], M[:, :, 7:]
            WE, wE = WE + sgn * (-z * 1j * k * A - cF), wE + sgn * (z * 1j / k) * phi
            WH, wH = WH + sgn * (cA - (1j * k / z) * Fm), wH + sgn * (1j / (k * z)) * psi
            E.append(-z * (1j * k * A + (1j / k) * gphi) - cF)
        loc = lambda s: self.rel[..., None] * self.a[s][:, None, None] - self.b[s][:, None]  # noqa: E731
        Js, M = loc(0) + loc(1), loc(2)
        n = self.normal[:, None, :, None].to(M.dtype).expand(-1, self.q, -1, M.shape[-1])
        t = lambda X_, V: torch.einsum("tkac,ta,tacb->tkb", X_.to(V.dtype), self.w.to(V.dtype), V)  # noqa: E731
        div = lambda v: (2 * self.cX)[..., None] * torch.einsum("ta,tab->tb", self.w.to(v.dtype), v)[:, None]  # noqa: E731
        v0, v1 = t(self.X, WE) + div(wE), t(self.X, WH) + div(wH)
        v2 = v1 - 0.5 * t(self.X, torch.linalg.cross(n, Js, dim=2)) - t(self.nX, sg * E[0]) - 0.5 * t(self.X, sg * M)
        v3 = t(self.X, Js) - t(self.X, sg * E[1]) - 0.5 * t(self.X, sg * torch.linalg.cross(n, M, dim=2))
        val = torch.stack([v0, v1, v2, v3], 2)  # (nt, k, type, B)
        y = torch.zeros(self.N + 1, X.shape[1], dtype=X.dtype, device=DEV)
        return y.index_add(0, self.row.reshape(-1), val.reshape(-1, X.shape[1]))[: self.N]

    def transpose(self, Y, sigma):
        """A^T Y, from the adjoint that autograd forms of the linear map."""
        x = torch.zeros_like(Y, requires_grad=True)
        y = self.apply(x, sigma)
        return torch.autograd.grad(y, x, Y.conj().resolve_conj())[0].conj().resolve_conj()

    def dense(self, sigma, step=48):
        A = torch.empty(self.N, self.N, dtype=torch.complex128, device=DEV)
        for i in range(0, self.N, step):
            m = min(step, self.N - i)
            U = torch.zeros(self.N, m, dtype=torch.complex128, device=DEV)
            U[i + torch.arange(m), torch.arange(m)] = 1
            A[:, i:i + m] = self.apply(U, sigma)
        return A

    # ---- conductivity, excitation, fields
    def sigma(self, kw):
        if "per_qpoint" in kw:
            return torch.as_tensor(kw["per_qpoint"], device=DEV)
        x = self.r[..., 0]
        if "bspline" in kw:
            x0, L, _, coef = kw["bspline"]
            return sum(float(cf) * self.bspline(i, len(coef), (x - x0) / L) for i, cf in enumerate(coef))
        out = torch.zeros_like(x)
        for x0, L, s0, d, _, sgn in kw["segments"]:
            out = out + s0 * (sgn * (x - x0) / L).clamp(0, 1) ** d
        return out

    @staticmethod
    def bspline(i, n, s):
        """Cubic basis function i of n on the clamped uniform knots of [0, 1] (Cox-de Boor)."""
        kn = [0.0] * 4 + [j / (n - 3) for j in range(1, n - 3)] + [1.0] * 4
        N = [((s >= kn[m]) & ((s < kn[m + 1]) | ((kn[m + 1] == 1.0) & (s <= 1.0)))).double() if kn[m] < kn[m + 1]
             else torch.zeros_like(s) for m in range(i, i + 4)]
        for d in range(1, 4):
            nxt = []
            for j, m in enumerate(range(i, i + 4 - d)):
                v = torch.zeros_like(s)
                if kn[m + d] > kn[m]:
                    v = v + (s - kn[m]) / (kn[m + d] - kn[m]) * N[j]
                if kn[m + d + 1] > kn[m + 1]:
                    v = v + (kn[m + d + 1] - s) / (kn[m + d + 1] - kn[m + 1]) * N[j + 1]
                nxt.append(v)
            N = nxt
        return N[0]

    def incident(self, src, r):
        """E and H of a complex-source-point beam in the interior medium at points r."""
        k, z = self.k[1], self.z[1]
        t = lambda v: torch.tensor(v, dtype=torch.complex128, device=DEV)  # noqa: E731
        p = t(src["pol"])
        D = r.to(torch.complex128) - (t(src["pos"]) - 1j * src["b"] * t(src["dir"]))
        R = (D * D).sum(-1).sqrt()
        Rh = D / R[..., None]
        G = torch.exp(-1j * k * R) / (4 * math.pi * R)
        u = 1j * k + 1 / R
        G1, G2 = -u * G, (u * u + 1 / R ** 2) * G
        rp = (Rh * p).sum(-1)
        hess = (G2 * rp)[..., None] * Rh + (G1 / R)[..., None] * (p - rp[..., None] * Rh)
        return -z * 1j * k * (G[..., None] * p + hess / k ** 2), torch.linalg.cross(G1[..., None] * Rh, p.expand_as(Rh))

    def rhs(self, srcs, sigma):
        sg, out = (sigma * ETA0)[..., None], []
        for s in srcs:
            E, H = self.incident(s, self.r)
            t = lambda V: torch.einsum("tkac,ta,tac->tk", self.X.to(V.dtype), self.w.to(V.dtype), V)  # noqa: E731
            e, h = t(E), t(H)
            val = torch.stack([e, h, h, t(sg * E)], 2)
            b = torch.zeros(self.N + 1, dtype=torch.complex128, device=DEV)
            out.append(b.index_add(0, self.row.reshape(-1), val.reshape(-1))[: self.N])
        return torch.stack(out, 1)

    def fields_at(self, x, pts, src):
        """Total interior E and H at points inside."""
        a, b = self.currents(x[:, None])
        J = (self.rel * a[1][:, :, None] - b[1][:, None, :, 0]) * self.w[..., None]
        M = -(self.rel * a[2][:, :, None] - b[2][:, None, :, 0]) * self.w[..., None]
        rJ, rM = 2 * a[1] * self.w, -2 * a[2] * self.w
        k, z, E, H = self.k[1], self.z[1], [], []
        J, M, rJ, rM, r = J.reshape(-1, 3), M.reshape(-1, 3), rJ.reshape(-1), rM.reshape(-1), self.r.reshape(-1, 3)
        for pt in torch.as_tensor(pts, device=DEV):
            D = pt - r
            R = D.norm(dim=1)
            G = torch.polar(1 / (4 * math.pi * R), -k * R)
            g = (-(1 / R + 1j * k) * G / R)[:, None] * D
            A, gp, cA = (G[:, None] * J).sum(0), (g * rJ[:, None]).sum(0), torch.linalg.cross(g, J).sum(0)
            F, gs, cF = (G[:, None] * M).sum(0), (g * rM[:, None]).sum(0), torch.linalg.cross(g, M).sum(0)
            E.append(-z * 1j * (k * A + gp / k) - cF)
            H.append(cA - 1j * (k * F + gs / k) / z)
        Ei, Hi = self.incident(src, torch.as_tensor(pts, device=DEV))
        return torch.stack(E) + Ei, torch.stack(H) + Hi


def _fit(E, t, betas):
    """{Re r, Im r, beta, residual, SWR, r_swr} of the two-wave fit with the smallest residual."""
    best = None
    for be in betas:
        M = np.stack([np.exp(-1j * be * t), np.exp(1j * be * t)], 1)
        g = M.conj().T @ M
        a, c = np.linalg.solve(g, M.conj().T @ E)
        res = np.linalg.norm(M @ [a, c] - E)
        if best is None or res < best[0]:
            best = (res, c / a, be)
    swr = np.abs(E).max() / np.abs(E).min()
    return np.array([[best[1].real, best[1].imag, best[2], best[0] / np.linalg.norm(E), swr, (swr - 1) / (swr + 1)]])


def exact(case, seed):
    c = case
    if c["mesh"] == "coupler" or (c["path"] in ("solve", "gradient") and c["nx"] * (c["ny"] + c["nz"]) > 600):
        return None
    R = _Reference(c)
    kw = _sigma(c, seed, R.nt, R.region)
    sigma = R.sigma(kw)
    srcs = _sources(c, seed) if c["mesh"] != "sphere" else []
    if c["path"] in ("apply", "adjoint", "sweep"):
        X = _vectors(seed, c["nrhs"], R.N, torch.complex64 if c["prec"] == 64 else torch.complex128)
        X = X.to(DEV).to(torch.complex128)
        f = R.transpose if c["path"] == "adjoint" else R.apply
        y = torch.stack([f(X[i][:, None], sigma)[:, 0] for i in range(c["nrhs"])])
        return [R.rhs(srcs, sigma).T.contiguous(), y] if c["path"] == "sweep" else y
    if c["path"] == "post":
        x = _vectors(seed, 1, R.N, torch.complex128)[0].to(DEV)
        probe, pts = _probe(c)
        t = np.linspace(probe["t0"], probe["t1"], probe["npts"])
        line = np.asarray(probe["p0"])[None] + t[:, None] * np.array([1.0, 0, 0])
        El = R.fields_at(x, line, srcs[0])[0][:, 1].cpu().numpy()
        E, H = R.fields_at(x, pts, srcs[0])
        return [_fit(El, t, np.linspace(probe["beta_lo"], probe["beta_hi"], probe["nbeta"])),
                E[None].cpu().numpy(), H[None].cpu().numpy()]
    b = R.rhs(srcs, sigma)
    A = R.dense(sigma)
    x = torch.linalg.solve(A, b)
    if c["path"] == "solve":
        return x.T.contiguous()
    # gradient of |f^T x|^2 with respect to the spline coefficients, by the adjoint system
    zero = torch.zeros_like(sigma)
    f = R.rhs([_receiver(c, seed)], zero)[:, 0]
    lam = torch.linalg.solve(A.T, 2 * f * torch.dot(f, x[:, 0]).conj())
    r0 = R.apply(x, zero) - R.rhs(srcs, zero)
    n, s, g = len(kw["bspline"][3]), (R.r[..., 0] - kw["bspline"][0]) / kw["bspline"][1], []
    for i in range(n):
        si = R.bspline(i, n, s)
        g.append(-float((lam @ (R.apply(x, si) - R.rhs(srcs, si) - r0)[:, 0]).real))
    return [x[:, 0].contiguous(), torch.tensor(g, dtype=torch.float64)]
