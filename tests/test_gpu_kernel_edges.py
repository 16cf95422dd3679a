"""Edge sizes of the kernels of a product, its set-up and its solves.

Forms that the workloads of the other files do not reach: meshes of one edge class, rows of the
near matrix with the self pair only, with every edge (a whole CTA per row, longer than the sorted
length) and between (a warp per row), odd and even boxes of active columns in the parity-split
(y, z) sums, every batch size (groups of one to four right-hand sides, full and ragged), a second
conductivity (the parts that depend on it are formed again), solves of one and eight right-hand
sides, and field points split over one and many CTAs.  Tolerances are those of the parity tests:
1e-10 in complex128 and 1e-5 in complex64 of the oracle's largest entry, 1e-12 and 1e-5 for the
dot-product identity of the transposed operator.
"""

import dataclasses

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import cases
import paper_1004_5076_gb300 as sc
import synth
from oracle import excitation, mesh, pfft, post

from test_gpu_adjoint import _dot_gap
from test_gpu_parity import TOL32, TOL64, build, gpu_apply

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _require_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _plate(name, region=None, **kw):
    c = cases.plate_thin()
    if region is not None:
        c.mesh = synth.Mesh(c.mesh.V, c.mesh.T, np.full(c.mesh.nt, region, np.int32))
    return dataclasses.replace(c, name=name, **kw)


def _box(name, ny, nz, padded, p, r_near):
    m = synth.waveguide(1.5, 0.3, 0.16, 9, ny, nz, 0.4, 0.3)
    return cases.Case(name, m, (4.0, 1.0, 1.5, 1.0, 1.3), synth.grid_for_mesh(m.V, padded, p=p), 3, r_near,
                      sigma_scale=0.002, seed=31, transverse="direct")


def _dense_rows():
    """1920 edges that are all near one another, on a few sampled rows."""
    m = synth.icosphere(3, 1.0)
    m = synth.Mesh(m.V, m.T, (m.V[m.T].mean(1)[:, 0] > 0.2).astype(np.int32))
    return cases.Case("dense_rows", m, (2.25, 1.0, 1.0, 1.0, 1.55), synth.grid_for_mesh(m.V, (16, 16, 16), p=2), 1,
                      100.0, sigma_scale=0.003, seed=32)


EDGES = [
    lambda: _plate("no_absorber", 0, sigma_scale=0.0),
    lambda: _plate("all_absorber", 1),
    lambda: _plate("self_pairs", r_near=1e-6),
    lambda: _plate("all_pairs", r_near=100.0),
    lambda: _box("box_p2", 4, 2, (16, 16, 8), 2, 0.25),
    lambda: _box("box_p3", 5, 3, (32, 16, 16), 3, 0.13),
    lambda: _box("box_p4", 3, 2, (32, 16, 16), 4, 0.1),
    _dense_rows,
]


@pytest.mark.parametrize("mk", EDGES, ids=lambda f: f().name)
def test_products_of_every_batch_size(mk):
    case = mk()
    mh, op, g, med, sig = build(case)
    U = np.stack([cases.synth.complex_normal(g.N, seed=40 + c) for c in range(2)])
    mix = cases.synth.complex_normal(16, seed=45).reshape(8, 2)  # eight columns, two oracle applies
    X = mix @ U
    if case.name == "dense_rows":
        edges = np.random.default_rng(3).choice(g.ne, 3, replace=False)
        targets = np.unique(g.edge_t[edges].reshape(-1))
        rows = mesh.row_index(g)[edges]
        rows = rows[rows >= 0]
        Y_or = pfft.PFFT(g, med, case.grid, case.r_near).apply(U.T, sig, targets=targets).T[:, rows]
    else:
        rows = np.arange(g.N)
        Y_or = pfft.PFFT(g, med, case.grid, case.r_near).apply(U.T, sig).T
    Y_or = mix @ Y_or
    for prec, dt, tol in ((sc.SCABEM_C128, torch.complex128, TOL64), (sc.SCABEM_C64, torch.complex64, TOL32)):
        for k in range(1, 9):
            x = torch.as_tensor(X[:k]).to(dt).cuda().contiguous()
            y = torch.empty_like(x)
            sc.scabem_apply(op, x, y, nrhs=k, ld=g.N, prec=prec)
            torch.cuda.synchronize()
            d = np.abs(y.cpu().numpy()[:, rows] - Y_or[:k])
            assert np.all(d.max(1) <= tol * np.abs(Y_or[:k]).max(1)), (prec, k)
        assert _dot_gap(op, g.N, prec, 50) < (1e-12 if prec == sc.SCABEM_C128 else 1e-5)


@pytest.mark.parametrize("mk", [cases.plate_thin, cases.guide_small], ids=lambda f: f.__name__)
@pytest.mark.parametrize("shift", [0, 3])
def test_transposed_product_in_place(mk, shift):
    case = mk()
    mh, op, g, med, sig = build(case)
    for dt, prec in ((torch.complex128, sc.SCABEM_C128), (torch.complex64, sc.SCABEM_C64)):
        v = torch.as_tensor(cases.synth.complex_normal(g.N + shift, seed=90)).to(dt).cuda()
        ref = torch.empty(g.N, dtype=dt, device="cuda")
        sc.scabem_apply_adjoint(op, v[:g.N].clone(), ref, prec=prec)
        sc.scabem_apply_adjoint(op, v[:g.N], v[shift:], prec=prec)  # overlapping by all but `shift` values
        torch.cuda.synchronize()
        assert torch.equal(v[shift:], ref)


def test_second_conductivity_equals_a_new_operator():
    case = cases.guide_short()
    m, x = case.mesh, None
    out = []
    for again in (False, True):
        mh = sc.scabem_mesh_create(m.V, m.T, m.region)
        op = sc.scabem_op_create(mh, case.media, case.grid.n, case.grid.h, case.grid.origin, case.grid.p, case.q,
                                 case.r_near, 3)
        g = mesh.build(m.V, m.T, m.region, q=case.q)
        sig = cases.sigma_points(case, g.qpts).reshape(-1)
        if again:
            sc.scabem_set_sigma(op, per_qpoint=3.0 * sig[::-1].copy())
        sc.scabem_set_sigma(op, per_qpoint=sig)
        if x is None:
            x = cases.synth.complex_normal(g.N, seed=60)
        b = torch.as_tensor(x).cuda()
        u = torch.zeros_like(b)
        info = sc.scabem_solve(op, b, u, tol=1e-4, restart=40, maxit=4000, refine_tol=1e-9, prec=sc.SCABEM_C64)
        torch.cuda.synchronize()
        assert info[0]["status"] == 0
        out.append([gpu_apply(op, x, sc.SCABEM_C128), gpu_apply(op, x, sc.SCABEM_C64), u.cpu().numpy()])
    for a, b in zip(*out):  # the same sums in the same order
        assert np.array_equal(a, b)


@pytest.mark.parametrize("nrhs", [1, 8])
def test_solves_of_one_and_eight(nrhs):
    case = cases.guide_small()
    mh, op, g, med, sig = build(case)
    b = torch.as_tensor(np.stack([cases.synth.complex_normal(g.N, seed=70 + c) for c in range(nrhs)])).cuda()
    x = torch.zeros_like(b)
    info = sc.scabem_solve(op, b, x, nrhs=nrhs, ld=g.N, tol=1e-4, restart=80, maxit=8000, refine_tol=1e-9,
                           prec=sc.SCABEM_C64)
    r = torch.empty_like(b)
    sc.scabem_apply(op, x, r, nrhs=nrhs, ld=g.N)
    torch.cuda.synchronize()
    for c in range(nrhs):
        assert info[c]["status"] == 0
        assert (b[c] - r[c]).norm() <= 1e-8 * b[c].norm()


@pytest.mark.parametrize("npts", [1, 33, 2500])
def test_field_points(npts):
    case = cases.sphere_mixed()
    mh, op, g, med, sig = build(case)
    x = cases.synth.complex_normal(g.N, seed=80) * 1e-2
    src = sc.make_source("beam", "i", pos=(0.1, 0, 0), dir=(1, 0, 0), pol=(0, 1, 0), b=0.3)
    pts = 0.3 * np.random.default_rng(5).uniform(-1.0, 1.0, (npts, 3))
    E = sc.scabem_fields(op, torch.as_tensor(x).cuda(), pts, inc=src)[0]
    at = np.unique(np.linspace(0, npts - 1, 40).astype(int))
    ki, zi = med.k[1], med.z[1]
    E_or = post.radiated(g, x, pts[at], ki, zi, "i") + excitation.beam(pts[at], ki, zi, (0.1, 0, 0), (1, 0, 0), 0.3,
                                                                       (0, 1, 0))[0]
    assert np.max(np.abs(E[at] - E_or)) <= 1e-10 * np.max(np.abs(E_or))
