"""Calls on a stream of the caller's own, beside work queued on the default stream.

A torch stream is not ordered with the default stream.  Every sum of the library runs in a fixed
order, so the results equal those on the default stream bit for bit.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import cases
import paper_1004_5076_gb300 as sc

from test_gpu_parity import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _require_gpu():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")


def _calls(op, N, nrhs, b, stream):
    """A solve and both products in both precisions, on `stream`."""
    with torch.cuda.stream(stream):
        x = torch.zeros_like(b)
        info = sc.scabem_solve(op, b, x, nrhs=nrhs, ld=N, tol=1e-4, restart=80, maxit=8000, refine_tol=1e-9,
                               prec=sc.SCABEM_C64)
        out = [x]
        for dt, prec in ((torch.complex128, sc.SCABEM_C128), (torch.complex64, sc.SCABEM_C64)):
            v = b.to(dt)
            for product in (sc.scabem_apply, sc.scabem_apply_adjoint):
                out.append(torch.empty_like(v))
                product(op, v, out[-1], nrhs=nrhs, ld=N, prec=prec)
        stream.synchronize()
    assert all(i["status"] == 0 for i in info)
    return out


def _busy():
    """About 0.1 s of ordinary work on the current stream."""
    a = torch.full((4096, 4096), 1e-4, device="cuda")
    torch.cuda.synchronize()
    for _ in range(40):
        a = a @ a


@pytest.mark.parametrize("nrhs", [1, 8])
def test_calls_on_another_stream(nrhs):
    mh, op, g, med, sig = build(cases.guide_small())
    b = torch.as_tensor(np.stack([cases.synth.complex_normal(g.N, seed=110 + c) for c in range(nrhs)])).cuda()
    ref = _calls(op, g.N, nrhs, b, torch.cuda.current_stream())
    own = torch.cuda.Stream()
    _busy()
    out = _calls(op, g.N, nrhs, b, own)
    torch.cuda.synchronize()
    for u, v in zip(out, ref):
        assert torch.equal(u, v)


def _create(case):
    m = case.mesh
    mh = sc.scabem_mesh_create(m.V, m.T, m.region)
    return sc.scabem_op_create(mh, case.media, case.grid.n, case.grid.h, case.grid.origin, case.grid.p, case.q,
                               case.r_near, 3), sc.scabem_mesh_info(mh)[2]


def test_operator_created_on_another_stream():
    """After an operator with another quadrature rule, whose points must not be met."""
    out = []
    for own in (None, torch.cuda.Stream()):
        _create(cases.plate_p4_q7())
        if own is not None:
            _busy()
        with torch.cuda.stream(own):
            op, N = _create(cases.plate_thin())
        x = torch.as_tensor(cases.synth.complex_normal(N, seed=120)).cuda()
        torch.cuda.synchronize()
        out.append(torch.empty_like(x))
        sc.scabem_apply(op, x, out[-1])
    torch.cuda.synchronize()
    assert torch.equal(out[0], out[1])
