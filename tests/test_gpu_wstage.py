"""The 81-point stencils around the line between the two ways they read W~: a
block's ring in shared memory wherever it fits, or each thread's own loads (one
right-hand side at N_c = 3 and 4; FP64 Laplacians; FP64 D_B with fewer than four
threads per site; N_c = 1 Laplacians on site-inner vectors).  Odd volumes leave a ragged last block whose idle threads still
take part in the copies; extent 2 wraps every offset."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import check, to_device, to_numpy
from paper_2112_14640_gb300 import dirac as D
from paper_2112_14640_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BC = (1, 1, -1, -1)


@pytest.mark.parametrize("nc,nv,prec,links", [
    (3, 1, D.F32, 0), (4, 1, D.F32, 0), (3, 1, D.F64, 0), (1, 8, D.F32, 0), (1, 24, D.F32, 0),
    (3, 3, D.F32, 0), (3, 4, D.F32, 0), (3, 7, D.F32, 0), (3, 8, D.F64, 0), (3, 64, D.F32, 0), (1, 5, D.F32, 0),
    (2, 6, D.F64, 0), (4, 4, D.F32, 0), (4, 5, D.F64, 0), (1, 16, D.BF16, 0), (2, 9, D.F16, 0), (3, 12, D.BF16, 0),
    (3, 16, D.F16, 1), (4, 8, D.F16, 0)])
@pytest.mark.parametrize("dims", [(3, 5, 2, 7), (2, 2, 2, 2)])
@pytest.mark.parametrize("kind", [D.BRILLOUIN, D.BLAP, D.BSUV])
def test_staged_and_direct_w(kind, dims, nc, nv, prec, links):
    """Default launch and every VR, both layouts, D and its dagger (the parity
    tolerances of the stencils: 1e-12, 1e-5, 1e-2)."""
    if kind != D.BRILLOUIN and prec in (D.BF16, D.F16):
        pytest.skip("the Laplace operators have no 16-bit storage")
    U = I.gauge_field(dims, nc, 0.4, 91)
    ref = O.Operator(kind, U, BC)
    src = I.source(dims, nc, nv, 92, staggered=kind == D.BSUV)
    want = [ref.apply(src, 0.2), ref.apply_dagger(src, 0.2) if kind == D.BRILLOUIN else ref.apply(src, 0.2)]
    for layout in (D.SITE_OUTER, D.SITE_INNER):
        op = D.DiracOp(kind, torch.from_numpy(U).cuda(), nv, BC, prec, layout=layout, link_storage=links)
        x = to_device(op, src)
        for vr in (0, 1, 2, 4):
            if vr and nv % vr:
                continue
            op.set_launch(vr)
            for dag in (False, True):
                check(to_numpy(op, op.apply(x, m0=0.2, dagger=dag)), want[dag], prec, kind, layout, vr, dag)
        op.close()
