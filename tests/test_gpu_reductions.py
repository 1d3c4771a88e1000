"""Reductions of FP32 and BF16 vectors whose column sums leave FP32's range:
products are exact and a thread's few of them are summed in FP32, but threads
are added up in FP64, so only a thread's own share has to stay below 3.4e38.

Tolerance: a thread's pair (sum, error) of n products is off by at most
n^2 2^-48 of the sum of |product| (n = 64 at most here: 1.5e-11); the dot product's
operands are parallel, so that this is its own magnitude too."""
import math

import numpy as np
import pytest
import torch

from helpers import to_device
from paper_2112_14640_gb300 import dirac as D
from paper_2112_14640_gb300 import inputs as I

pytestmark = pytest.mark.gpu

DIMS = (8, 8, 8, 8)


def columns(op, v):
    """The stored vector as float64, (nv, everything else, re/im)."""
    c = torch.view_as_real(op.to_complex(v).to(torch.complex128))
    return np.moveaxis(c.reshape(-1, op.nv, 2).cpu().numpy(), 1, 0)


@pytest.mark.parametrize("prec", [D.F32, D.BF16])
@pytest.mark.parametrize("nv,layout", [(1, D.SITE_OUTER), (3, D.SITE_INNER), (12, D.SITE_OUTER), (64, D.SITE_INNER)])
def test_sums_past_the_range_of_fp32(prec, nv, layout):
    U = torch.from_numpy(I.gauge_field(DIMS, 3, 0.4, 31)).cuda()
    op = D.DiracOp(D.WILSON, U, nv, prec=prec, layout=layout)
    scale = 1e18   # 98304 components a column: |v|^2 about 1e41
    u = to_device(op, scale * I.source(DIMS, 3, nv, 32))
    x = columns(op, u)
    exact = np.array([math.fsum((x[v] ** 2).ravel()) for v in range(nv)])
    assert exact.min() > 3.4e38
    assert np.abs(op.norm2(u).cpu().numpy() / exact - 1).max() <= 1.5e-11
    dot = op.dot(u, u).cpu().numpy()
    assert np.abs(dot.real / exact - 1).max() <= 1.5e-11 and np.abs(dot.imag / exact).max() <= 1.5e-11
    # half of the sites: every second time slice would overflow on its own as well
    sites = math.prod(DIMS) // 2
    part = op.norm2_range(u, sites, sites).cpu().numpy() + op.norm2_range(u, 0, sites).cpu().numpy()
    assert np.abs(part / exact - 1).max() <= 3e-11
    part = op.dot_range(u, u, sites, sites).cpu().numpy().real + op.dot_range(u, u, 0, sites).cpu().numpy().real
    assert np.abs(part / exact - 1).max() <= 3e-11
    op.close()


def test_solves_past_the_range_of_fp32():
    """CG of a right-hand side whose |D^dag b|^2 is past FP32's range."""
    U = torch.from_numpy(I.gauge_field(DIMS, 3, 0.4, 33)).cuda()
    for layout in (D.SITE_OUTER, D.SITE_INNER):
        op = D.DiracOp(D.STAGGERED, U, 3, (1, 1, 1, -1), D.F32, layout=layout)
        b = to_device(op, 1e18 * I.source(DIMS, 3, 3, 34, staggered=True))
        x, st = op.solve(b, m0=0.5, tol=1e-5, maxit=500)
        assert st["status"] == 0 and max(st["relres"]) <= 1e-5, st
        xs, stats, rc = D.solve_batched([op], [b], m0s=[0.5], tol=1e-5, maxit=500)
        assert rc == 0 and stats[0]["iters"] > 0 and max(stats[0]["relres"]) <= 1e-5, stats
        assert float((xs[0] - x).abs().max()) <= 1e-3 * float(x.abs().max())
        op.close()
