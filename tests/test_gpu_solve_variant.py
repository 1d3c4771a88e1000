"""The launch variant of a site-outer operator reaches its solves, which iterate
on site-inner vectors.  In FP64 on a small lattice the variant shows in the
bits: without one the hops of a site are spread over lanes, with one the plain
kernel runs, and the two round differently."""
import pytest
import torch

from helpers import to_device
from paper_2112_14640_gb300 import dirac as D
from paper_2112_14640_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def solutions(op, b):
    kw = dict(m0=0.3, tol=1e-10, maxit=500)
    x, st = op.solve(b, **kw)
    (y,), (sb,), rc = D.solve_batched([op], [b], m0s=[0.3], tol=1e-10, maxit=500)
    assert st["status"] == 0 and rc == 0 and sb["status"] == 0
    return op.to_site_outer(x), op.to_site_outer(y)


@pytest.mark.parametrize("solver", [0, 1])   # dirac_solve, dirac_solve_batched
def test_set_launch_reaches_the_solves_of_a_site_outer_operator(solver):
    dims, nv = (4, 4, 2, 6), 4
    U = torch.from_numpy(I.gauge_field(dims, 3, 0.4, 81)).cuda()
    src = I.source(dims, 3, nv, 82)
    got = {}
    for layout in (D.SITE_OUTER, D.SITE_INNER):
        op = D.DiracOp(D.WILSON, U, nv, (1, 1, 1, -1), D.F64, layout=layout)
        b = to_device(op, src)
        got[layout, "split"] = solutions(op, b)[solver]
        op.set_launch(2, 3, 256)
        got[layout, "plain"] = solutions(op, b)[solver]
        op.set_launch(0)
        got[layout, "default"] = solutions(op, b)[solver]
        op.close()
    for variant in ("split", "plain", "default"):
        assert torch.equal(got[D.SITE_OUTER, variant], got[D.SITE_INNER, variant]), variant
    assert not torch.equal(got[D.SITE_INNER, "plain"], got[D.SITE_INNER, "split"])
    assert torch.equal(got[D.SITE_INNER, "default"], got[D.SITE_INNER, "split"])
