"""The D_W and D_S force against the oracle at every number of right-hand sides
a load can take (1, 2, 4 and remainders), on vectors that start on a 16-byte but
not a 32-byte boundary, and at N_c 1..8.  Tolerance: a component is a sum of
8 N_v products (N_v = 12: 96) of rounded inputs, FP32 unit roundoff 6e-8: 1e-5."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import rel_l2, to_device
from paper_2112_14640_gb300 import dirac as D
from paper_2112_14640_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BC = (1, -1, 1, -1)


def shifted(v):
    """The same vector 16 bytes past a 32-byte boundary."""
    n = v.numel() * v.element_size()
    raw = torch.empty(n + 64, dtype=torch.uint8, device=v.device)
    at = (-raw.data_ptr()) % 32 + 16
    out = raw[at:at + n].view(v.dtype).view(v.shape)
    out.copy_(v)
    return out


@pytest.mark.parametrize("kind", [D.WILSON, D.STAGGERED])
@pytest.mark.parametrize("nc,nv", [(3, 1), (3, 2), (3, 6), (3, 8), (3, 12), (1, 4), (2, 8), (4, 4), (4, 2), (5, 4), (6, 2), (7, 2),
                                   (8, 1), (8, 3)])
def test_force_widths(kind, nc, nv):
    dims = (2, 4, 2, 6)
    U = I.gauge_field(dims, nc, 0.4, 71)
    psi = I.source(dims, nc, nv, 72, staggered=kind == D.STAGGERED)
    chi = I.source(dims, nc, nv, 73, staggered=kind == D.STAGGERED)
    ref = O.Operator(kind, U, BC)
    force, grad = ((O.wilson_force, O.wilson_action_gradient) if kind == D.WILSON
                   else (O.staggered_force, O.staggered_action_gradient))
    want = force(ref, psi, chi), grad(ref, psi, chi)
    for prec, tol in ((D.F64, 1e-12), (D.F32, 1e-5)):
        for layout in (D.SITE_OUTER, D.SITE_INNER):
            op = D.DiracOp(kind, torch.from_numpy(U).cuda(), nv, BC, prec, layout=layout)
            x, y = to_device(op, psi), to_device(op, chi)
            for a, b in ((x, y), (shifted(x), y), (x, shifted(y))):
                for mode, w in ((D.FORCE_TA, want[0]), (D.FORCE_GRAD, want[1])):
                    got = op.force(a, b, mode).to(torch.complex128).cpu().numpy()
                    assert rel_l2(got, w) <= tol, (prec, layout, mode)
            op.close()
