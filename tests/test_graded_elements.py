"""mu303 with W = I where the fixed-point kernels' numbers have to span a range.

Elements whose size varies inside the element: a point
whose T is r times smaller than the element's largest one. In FP64 the map's
own rounding leaves T there with a relative error of some 8 eps r (sums of at
most 5 products per direction), of which det T and P take a few: 100 eps r for
each quantity (normwise for the nodal ones, which the small points dominate as
P grows as 1 / |T|).

Meshes within a relative distance d of the ideal one, where the terms of P
cancel to d of their size: in FP64 what is left has an error of some tenths of
eps / d (the oracle's, against its formulas in extended precision): 10 eps / d."""
import numpy as np
import pytest

import oracle
from paper_1807_09807_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu

M = np.array([[1.0, 0.2, -0.1], [0.05, 0.9, 0.15], [-0.2, 0.1, 1.1]])


def graded(order, nq, ratio, nx=(1, 1, 1)):
    """Elements drawn together towards their corner (0, 0, 0) by the quadratic or
    cubic whose slope varies by about `ratio` along an axis, then sheared."""
    x, en, fx = mg.structured(3, order, nx)
    p = 1 if order == 2 else 2
    a = 1.0 / (ratio ** (1.0 / p) - 1.0) if ratio > 1 else 1e9
    if ratio > 1:
        x = ((x + a) ** (p + 1) - a ** (p + 1)) / ((1 + a) ** (p + 1) - a ** (p + 1))
    x = np.ascontiguousarray(M @ x)
    return mg.Mesh(dim=3, order=order, nx=nx, x=x, x_ideal=x, elem_nodes=en, fixed=np.zeros_like(fx), nq=nq,
                   quad_kind=mg.GLL if nq == order + 1 else mg.GL, metric=303)


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("order,nq", [(2, 3), (2, 4), (3, 4), (3, 5), (4, 5), (4, 6)])   # GLL (points at the corners), GL
@pytest.mark.parametrize("ratio", [1, 10, 100])
def test_sizes_that_vary_inside_an_element(order, nq, ratio):
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = graded(order, nq, ratio)
    orc = oracle.Problem(3, order, m.elem_nodes, m.nnode, m.fixed, nq, 303, quad_kind=m.quad_kind)
    ctx = tm.Context.from_mesh(m)
    A = orc.jacobians(m.x).reshape(-1, 9)
    r = np.abs(A).max() / np.abs(A).max(axis=1).min()
    tol = 100 * 2.2e-16 * max(r, 1.0)
    x, v = torch.tensor(m.x, device="cuda"), np.random.default_rng(1).standard_normal(m.x.shape)
    vd = torch.tensor(v, device="cuda")
    Fo, go, yo = orc.energy(m.x), orc.gradient(m.x), orc.hess_apply(m.x, v)
    F = ctx.energy(x)
    assert F[0] == Fo[0] == tm.OK
    assert abs(F[2] - Fo[2]) <= tol * Fo[2] and abs(F[1] - Fo[1]) <= tol * Fo[1]
    assert abs(ctx.element_min_detA(x).item() - Fo[2]) <= tol * Fo[2]
    assert rel(ctx.gradient(x).cpu().numpy(), go) <= tol
    assert rel(ctx.hess_apply(x, vd).cpu().numpy(), yo) <= tol
    g, y = ctx.gradient_hess_apply(x, vd)
    assert rel(g.cpu().numpy(), go) <= tol and rel(y.cpu().numpy(), yo) <= tol
    g, F2, md = ctx.energy_gradient(x)
    assert rel(g.cpu().numpy(), go) <= tol and abs(F2.item() - Fo[1]) <= tol * Fo[1]
    assert abs(md.item() - Fo[2]) <= tol * Fo[2]


@pytest.mark.parametrize("order,nq", [(1, 2), (2, 4), (3, 5), (4, 6)])
@pytest.mark.parametrize("d", [1e-6, 1e-8, 1e-9, 1e-10])
def test_terms_that_cancel(order, nq, d):
    """The gradient a distance d from a uniform mesh, and the Hessian action
    there on a direction as close to x itself (P is homogeneous in T, so both
    are of order d)."""
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    x, en, fx = mg.structured(3, order, (2, 2, 2))
    rng = np.random.default_rng(4)
    v = x + d * rng.standard_normal(x.shape)
    x = x + d * rng.standard_normal(x.shape)
    fx = np.zeros_like(fx)
    orc = oracle.Problem(3, order, en, x.shape[1], fx, nq, 303)
    ctx = tm.Context(3, order, x.shape[1], None, fx, nq, 303, structured=[2, 2, 2], nelem=8)
    xd, vd = torch.tensor(x, device="cuda"), torch.tensor(v, device="cuda")
    tol = 10 * 2.2e-16 / d
    go, yo = orc.gradient(x), orc.hess_apply(x, v)
    assert rel(ctx.gradient(xd).cpu().numpy(), go) <= tol and rel(ctx.hess_apply(xd, vd).cpu().numpy(), yo) <= tol
    g, y = ctx.gradient_hess_apply(xd, vd)
    assert rel(g.cpu().numpy(), go) <= tol and rel(y.cpu().numpy(), yo) <= tol
    assert rel(ctx.energy_gradient(xd)[0].cpu().numpy(), go) <= tol
    ctx.linearize(xd)
    assert rel(ctx.hess_apply_pa(vd).cpu().numpy(), yo) <= tol
