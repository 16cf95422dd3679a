"""Forward products whose result overlaps their input.

The rows of a product gather x while others already write y, so an overlapping x is copied first.
One column may overlap y in any way; of nine columns, which go as eight and one, y is x itself.  The
result equals that of separate buffers bit for bit.
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


@pytest.mark.parametrize("mk", [cases.plate_thin, cases.guide_small], ids=lambda f: f.__name__)
@pytest.mark.parametrize("prec,dt", [(sc.SCABEM_C128, torch.complex128), (sc.SCABEM_C64, torch.complex64)],
                         ids=["c128", "c64"])
def test_forward_product_in_place(mk, prec, dt):
    mh, op, g, med, sig = build(mk())
    for shift in (0, 3):
        v = torch.as_tensor(cases.synth.complex_normal(g.N + shift, seed=130)).to(dt).cuda()
        ref = torch.empty(g.N, dtype=dt, device="cuda")
        sc.scabem_apply(op, v[:g.N].clone(), ref, prec=prec)
        sc.scabem_apply(op, v[:g.N], v[shift:], prec=prec)
        torch.cuda.synchronize()
        assert torch.equal(v[shift:], ref), shift
    x = torch.as_tensor(np.stack([cases.synth.complex_normal(g.N, seed=140 + c) for c in range(9)])).to(dt).cuda()
    ref = torch.empty_like(x)
    sc.scabem_apply(op, x.clone(), ref, nrhs=9, ld=g.N, prec=prec)
    sc.scabem_apply(op, x, x, nrhs=9, ld=g.N, prec=prec)
    torch.cuda.synchronize()
    assert torch.equal(x, ref)
