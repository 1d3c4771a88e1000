"""FP64 applies on lattices small enough for a site's hops to be spread over
lanes, against the oracle: every kind, N_c 1..4, odd and wrapping extents, one
to many right-hand sides, both layouts, daggers; and the line above which the
plain kernels run (9728 sites times RHS), on both sides of it."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import check, to_device, to_numpy
from paper_2112_14640_gb300 import dirac as D
from paper_2112_14640_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BC = (1, -1, 1, -1)
KINDS = [D.WILSON, D.BRILLOUIN, D.STAGGERED, D.WLAP, D.BLAP, D.WSUV, D.BSUV]


@pytest.mark.parametrize("dims,nc,nv", [((2, 2, 2, 2), 3, 1), ((3, 5, 2, 3), 1, 3), ((3, 2, 5, 4), 2, 7),
                                        ((4, 2, 6, 2), 4, 2), ((5, 3, 3, 7), 3, 5)])
@pytest.mark.parametrize("kind", KINDS)
def test_split_applies(kind, dims, nc, nv):
    if kind == D.STAGGERED:
        dims = tuple(d + (d & 1) for d in dims)
    U = I.gauge_field(dims, nc, 0.4, 95)
    colour_only = kind in (D.STAGGERED, D.WSUV, D.BSUV)
    src = I.source(dims, nc, nv, 96, staggered=colour_only)
    ref = O.Operator(kind, U, BC)
    dagger = (lambda v: ref.apply_dagger(v, 0.3)) if kind in (D.WILSON, D.BRILLOUIN, D.STAGGERED) else None
    for layout in (D.SITE_OUTER, D.SITE_INNER):
        op = D.DiracOp(kind, torch.from_numpy(U).cuda(), nv, BC, D.F64, layout=layout)
        x = to_device(op, src)
        check(to_numpy(op, op.apply(x, m0=0.3)), ref.apply(src, 0.3), D.F64, kind, layout)
        if dagger:
            check(to_numpy(op, op.apply(x, m0=0.3, dagger=True)), dagger(src), D.F64, kind, layout, "dagger")
        op.close()


@pytest.mark.parametrize("kind", [D.WILSON, D.STAGGERED, D.BRILLOUIN, D.BLAP])
@pytest.mark.parametrize("dims,nv", [((8, 4, 4, 2), 37), ((8, 4, 4, 2), 38)])   # 9472, 9728 items
def test_both_sides_of_the_line(kind, dims, nv):
    """Below the line the hops are spread over lanes, so the result differs in
    its last bits from the plain kernel's, which a chosen variant launches; on
    it the two are the same kernel."""
    U = I.gauge_field(dims, 3, 0.4, 97)
    src = I.source(dims, 3, nv, 98, staggered=kind == D.STAGGERED)
    op = D.DiracOp(kind, torch.from_numpy(U).cuda(), nv, BC, D.F64, layout=D.SITE_INNER)
    x = to_device(op, src)
    out = op.apply(x, m0=0.3)
    check(to_numpy(op, out), O.Operator(kind, U, BC).apply(src, 0.3), D.F64, kind, dims, nv)
    op.set_launch(1)
    split = np.prod(dims) * nv < 9728
    assert torch.equal(op.apply(x, m0=0.3), out) != split
    op.close()


def test_a_chosen_variant_is_the_plain_kernel_and_tuning_keeps_the_split_one():
    dims, nv = (4, 4, 2, 6), 4
    U = I.gauge_field(dims, 3, 0.4, 93)
    src = I.source(dims, 3, nv, 94)
    ref = O.Operator(D.WILSON, U, BC).apply(src, 0.2)
    op = D.DiracOp(D.WILSON, torch.from_numpy(U).cuda(), nv, BC, D.F64)
    x = to_device(op, src)
    split = op.apply(x, m0=0.2)
    op.set_launch(2, 3, 256)
    check(to_numpy(op, op.apply(x, m0=0.2)), ref, D.F64, "plain")
    op.autotune(0.2)
    assert torch.equal(op.apply(x, m0=0.2), split)
    op.close()


def test_parts_of_a_lattice_give_the_same_bits():
    """A range of output sites takes the same kernel as the whole lattice."""
    dims, nv = (4, 4, 2, 6), 3
    U = I.gauge_field(dims, 3, 0.4, 99)
    op = D.DiracOp(D.WILSON, torch.from_numpy(U).cuda(), nv, BC, D.F64)
    x = to_device(op, I.source(dims, 3, nv, 100))
    whole = op.apply(x, m0=0.1)
    part = torch.zeros_like(x)
    op.apply_range(x, part, 32, 64, m0=0.1)
    assert torch.equal(part[1:3], whole[1:3]) and torch.count_nonzero(part[0]) == 0
    assert torch.count_nonzero(part[3:]) == 0
    op.close()
