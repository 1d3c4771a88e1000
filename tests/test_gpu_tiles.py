"""The site-tiled W builder at the edges of its
tiles: volumes that are no multiple of a tile, lattices smaller than one
tile, extents of 2 and 3 (every offset wraps), every N_c and storage the tile
size depends on."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import rel_l2
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
