"""CG's runs of iterations enqueued ahead of the host: run lengths that are no
multiple of a graph's iterations, iteration limits inside a run, recompute
intervals of every size, one to 64 right-hand sides on lattices smaller than
one reduction block; and the site-inner order the iteration runs in, which a
site-outer operator must not show."""
import numpy as np
import pytest
import torch

import oracle as O
from helpers import to_device, to_numpy
from paper_2112_14640_gb300 import dirac as D
from paper_2112_14640_gb300 import inputs as I

pytestmark = pytest.mark.gpu

BC = (1, 1, 1, -1)


def problem(kind, dims, nv, prec, layout, seed=61):
    U = I.gauge_field(dims, 3, 0.4, seed)
    op = D.DiracOp(kind, torch.from_numpy(U).cuda(), nv, BC, prec, layout=layout)
    b = I.source(dims, 3, nv, seed + 1, staggered=kind == D.STAGGERED)
    return op, O.Operator(kind, U, BC), b


def relres(ref, x, b, m0):
    bN = ref.apply_dagger(b, m0)
    return np.sqrt(O.norm2(bN - ref.apply_normal(x, m0)) / O.norm2(bN))


@pytest.mark.parametrize("every", [0, 1, 7, 23])
@pytest.mark.parametrize("kind,dims,nv", [(D.STAGGERED, (2, 2, 2, 2), 1), (D.STAGGERED, (4, 2, 4, 6), 64),
                                          (D.WILSON, (3, 2, 3, 5), 17)])
def test_recompute_intervals(kind, dims, nv, every):
    m0 = 0.2
    op, ref, b = problem(kind, dims, nv, D.F64, D.SITE_OUTER)
    x, st = op.solve(to_device(op, b), m0=m0, tol=1e-10, maxit=4000, recompute_every=every)
    assert st["status"] == 0 and st["recomputes"] >= 1
    assert np.all(relres(ref, to_numpy(op, x), b, m0) < 1.01e-10)
    op.close()


@pytest.mark.parametrize("maxit", [1, 4, 5, 6, 13])
@pytest.mark.parametrize("inner", [D.F64, D.F32])
def test_iteration_limit_inside_a_run(inner, maxit):
    """The solver stops after exactly maxit iterations and its residual is the
    one the oracle finds (FP64 outer residuals: 1e-3 relative)."""
    m0 = 0.05
    op, ref, b = problem(D.STAGGERED, (4, 4, 4, 6), 3, D.F64, D.SITE_OUTER)
    x, st = op.solve(to_device(op, b), m0=m0, tol=1e-10, maxit=maxit, inner_prec=inner)
    assert st["status"] == 1 and st["iters"] == maxit
    assert np.allclose(relres(ref, to_numpy(op, x), b, m0), st["relres"], rtol=1e-3)
    op.close()


@pytest.mark.parametrize("solver", [D.CG_NORMAL, D.CG_HPD, D.BICGSTAB])
@pytest.mark.parametrize("kind", [D.WILSON, D.STAGGERED])
@pytest.mark.parametrize("prec", [D.F64, D.F32])
def test_layouts_give_the_same_solution(prec, kind, solver):
    """Both layouts iterate on the same site-inner vectors: same bits, from a
    nonzero initial guess too."""
    if kind == D.STAGGERED and solver == D.BICGSTAB:
        pytest.skip("D_S is solved through the normal equations")
    xs = []
    for layout in (D.SITE_OUTER, D.SITE_INNER):
        op, ref, b = problem(kind, (4, 6, 2, 4), 5, prec, layout)
        x0 = to_device(op, I.source((4, 6, 2, 4), 3, 5, 77, staggered=kind == D.STAGGERED))
        x, st = op.solve(to_device(op, b), x=x0, m0=0.3, tol=1e-5, maxit=2000, solver=solver)
        assert st["status"] == 0
        y, stb, rc = D.solve_batched([op], [to_device(op, b)], m0s=[0.3], tol=1e-5, maxit=2000)
        assert rc == 0
        xs.append((to_numpy(op, x), to_numpy(op, y[0]), st["iters"]))
        op.close()
    assert np.array_equal(xs[0][0], xs[1][0]) and np.array_equal(xs[0][1], xs[1][1]) and xs[0][2] == xs[1][2]
