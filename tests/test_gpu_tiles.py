"""The site-tiled link kernels (W builder, Brillouin force) at the edges of
their tiles: volumes that are no multiple of a tile, lattices smaller than one
tile, extents of 2 and 3 (every offset wraps), every N_c and storage the tile
size depends on."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import rel_l2, to_device
from paper_2112_14640_gb300 import dirac as D
from paper_2112_14640_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BC = (1, -1, 1, -1)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 5, 2, 3), (7, 3, 2, 5)])
@pytest.mark.parametrize("nc,prec", [(1, D.F32), (2, D.F64), (3, D.F64), (3, D.F32), (3, D.BF16), (4, D.F64),
                                     (4, D.F32), (4, D.F16), (5, D.F32), (6, D.F64), (8, D.F64), (8, D.F32)])
def test_w_builder_tiles(nc, prec, dims):
    """W against the oracle's path enumeration: FP64 to 1e-13, FP32 to 1e-6
    (four levels of FP32 roundings), 16-bit links to their own rounding (FP32
    arithmetic from the caller's links, rounded twice: stored scaled, read
    back unscaled)."""
    U = I.gauge_field(dims, nc, 0.4, 81)
    op = D.DiracOp(D.BRILLOUIN, torch.from_numpy(U).cuda(), 1, BC, prec)
    got = op.to_complex(op.copy_w()).to(torch.complex128).cpu().numpy()
    want = np.delete(O.Operator(D.BRILLOUIN, U, BC).W, 40, axis=4)
    assert rel_l2(got, want) <= {D.F64: 1e-13, D.F32: 1e-6, D.BF16: 2.0 ** -8, D.F16: 2.0 ** -11}[prec]
    op.close()


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 5, 2, 3), (7, 3, 2, 5)])
@pytest.mark.parametrize("nc,nv,prec", [(1, 13, D.F32), (2, 1, D.F64), (3, 5, D.F64), (3, 40, D.F64), (3, 2, D.F32),
                                        (4, 3, D.F64), (4, 1, D.F32), (5, 2, D.F64)])
def test_brillouin_force_tiles(nc, nv, prec, dims):
    """The Brillouin force against the oracle's, both modes and layouts; 13 and
    40 RHS need more than one pass over the staged right-hand sides (12 N_c per
    pass).  FP64 to 1e-11, FP32 to 1e-5 (as the force tests)."""
    U = I.gauge_field(dims, nc, 0.4, 83)
    ref = O.Operator(D.BRILLOUIN, U, BC)
    psi, chi = I.source(dims, nc, nv, 84), I.source(dims, nc, nv, 85)
    want_f, want_g = O.brillouin_force(ref, psi, chi), O.brillouin_action_gradient(ref, psi, chi)
    for layout in (D.SITE_OUTER, D.SITE_INNER):
        op = D.DiracOp(D.BRILLOUIN, torch.from_numpy(U).cuda(), nv, BC, prec, layout=layout)
        p, c = to_device(op, psi), to_device(op, chi)
        tol = 1e-11 if prec == D.F64 else 1e-5
        got = op.force(p, c, D.FORCE_GRAD).to(torch.complex128).cpu().numpy()
        assert rel_l2(got, want_g) <= tol
        if nc > 1:   # su(1) has no traceless part
            got = op.force(p, c, D.FORCE_TA).to(torch.complex128).cpu().numpy()
            assert rel_l2(got, want_f) <= tol
        op.close()
