"""Vectors are only required to start on 16 bytes; groups of right-hand sides
wider than that are read 32 bytes at a time and need more, so a launch on less
aligned vectors takes narrower groups.  And launch variants of the N_c that
have one register class only."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import check, to_device, to_numpy
from paper_2112_14640_gb300 import dirac as D
from paper_2112_14640_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BC = (1, 1, 1, -1)


def shifted(v, nbytes):
    """A copy of v that starts nbytes past a 256-byte boundary."""
    buf = torch.zeros(v.numel() * v.element_size() + 512, dtype=torch.uint8, device=v.device)
    at = buf[nbytes:nbytes + v.numel() * v.element_size()].view(v.dtype).view(v.shape)
    at.copy_(v)
    assert at.data_ptr() % 256 == nbytes
    return at


@pytest.mark.parametrize("kind", [D.STAGGERED, D.WILSON, D.BRILLOUIN, D.WSUV])
@pytest.mark.parametrize("prec,vr", [(D.F32, 4), (D.F64, 2), (D.F64, 4), (D.F32, 0)])
def test_16_byte_aligned_vectors(kind, prec, vr):
    dims = (4, 2, 4, 6)
    U = I.gauge_field(dims, 3, 0.4, 71)
    src = I.source(dims, 3, 8, 72, staggered=kind in (D.STAGGERED, D.WSUV))
    ref = O.Operator(kind, U, BC)
    op = D.DiracOp(kind, torch.from_numpy(U).cuda(), 8, BC, prec, layout=D.SITE_INNER)
    op.set_launch(vr)
    x = to_device(op, src)
    for a, b in ((16, 0), (0, 16), (48, 16), (32, 64)):
        xi, out = shifted(x, a), shifted(torch.zeros_like(x), b)
        op.apply(xi, out, m0=0.2)
        check(to_numpy(op, out), ref.apply(src, 0.2), prec, kind, vr, a, b)
    op.close()


@pytest.mark.parametrize("nc", [1, 2, 4, 5])
@pytest.mark.parametrize("kind", [D.WILSON, D.STAGGERED, D.WLAP, D.BSUV])
def test_other_colours_every_vr(kind, nc):
    """N_c without register classes, every VR."""
    dims = (4, 2, 2, 6)
    U = I.gauge_field(dims, nc, 0.4, 73)
    src = I.source(dims, nc, 4, 74, staggered=kind in (D.STAGGERED, D.BSUV))
    ref = O.Operator(kind, U, BC)
    for layout in (D.SITE_OUTER, D.SITE_INNER):
        op = D.DiracOp(kind, torch.from_numpy(U).cuda(), 4, BC, D.F32, layout=layout)
        x = to_device(op, src)
        for vr in (0, 1, 2, 4):
            if vr > 1 and nc > 4:
                continue
            op.set_launch(vr)
            check(to_numpy(op, op.apply(x, m0=0.2)), ref.apply(src, 0.2), D.F32, kind, nc, vr, layout)
        op.close()
