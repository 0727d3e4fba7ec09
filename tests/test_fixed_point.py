"""The FP64 element kernels contract in 64-bit fixed point with one exponent per
element and component: where that can go wrong. Against the oracle, whose sums
are plain FP64; its own A has a relative error of about eps |x| / h (2e-16
times ~10 here) per term, a metric adds a few digits, and 1e-11 leaves two
more (the components are compared one by one)."""
import numpy as np
import pytest

import oracle
from paper_1807_09807_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu

CASES = [(2, 1, 2, 2), (2, 2, 5, 2), (2, 3, 4, 9), (2, 4, 6, 2), (3, 1, 3, 303), (3, 2, 4, 302), (3, 3, 5, 303),
         (3, 4, 6, 303)]


def _mesh(dim, order, nq, metric, kind=mg.GL):
    nx = (3, 2) if dim == 2 else (3, 2, 2)
    x, en, fx = mg.structured(dim, order, nx)
    x = mg.jitter(x, fx, 0.08 / (order * 3), 5)
    return mg.Mesh(dim=dim, order=order, nx=nx, x=x, x_ideal=x, elem_nodes=en, fixed=fx, nq=nq, quad_kind=kind,
                   metric=metric)


def _per_component(a, b):
    return max(np.linalg.norm(a[c] - b[c]) / np.linalg.norm(b[c]) for c in range(a.shape[0]))


@pytest.mark.parametrize("dim,order,nq,metric", CASES)
def test_components_of_different_magnitude(dim, order, nq, metric):
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = _mesh(dim, order, nq, metric)
    m.x = np.ascontiguousarray(m.x * np.array([1.0, 1e-3, 30.0])[:dim, None])
    v = np.random.default_rng(1).standard_normal(m.x.shape) * np.array([1.0, 1e-3, 30.0])[:dim, None]
    ctx = tm.Context.from_mesh(m)
    orc = oracle.Problem(m.dim, m.order, m.elem_nodes, m.nnode, m.fixed, m.nq, m.metric)
    x = torch.tensor(m.x, device="cuda")
    g, y = ctx.gradient_hess_apply(x, torch.tensor(v, device="cuda"))
    assert _per_component(g.cpu().numpy(), orc.gradient(m.x)) < 1e-11
    assert _per_component(y.cpu().numpy(), orc.hess_apply(m.x, v)) < 1e-11
    ctx.linearize(x)
    y = ctx.hess_apply_pa(torch.tensor(v, device="cuda")).cpu().numpy()
    assert _per_component(y, orc.hess_apply(m.x, v)) < 1e-11


@pytest.mark.parametrize("dim,order,nq,metric", CASES)
def test_directions_of_any_exponent(dim, order, nq, metric):
    """A direction times a power of two: the same integers, so the same digits
    (near the ends of the exponent range another conversion rounds the last
    one: 1e-14 over the sums)."""
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = _mesh(dim, order, nq, metric)
    ctx = tm.Context.from_mesh(m)
    ctx.set_deterministic(True)
    x = torch.tensor(m.x, device="cuda")
    v = torch.tensor(np.random.default_rng(2).standard_normal(m.x.shape), device="cuda")
    y = ctx.hess_apply(x, v)
    for k in (-600, -40, 40, 600):
        assert torch.equal(ctx.hess_apply(x, v * 2.0 ** k), y * 2.0 ** k)
    for k in (-920, 920):
        assert (ctx.hess_apply(x, v * 2.0 ** k) * 2.0 ** -k - y).norm() < 1e-14 * y.norm()
    assert not ctx.hess_apply(x, torch.zeros_like(v)).any()


@pytest.mark.parametrize("dim,order,nq,metric", CASES)
@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
def test_a_value_that_is_not_finite_spoils_its_elements_only(dim, order, nq, metric, bad):
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = _mesh(dim, order, nq, metric)
    ctx = tm.Context.from_mesh(m)
    ctx.set_deterministic(True)
    x = torch.tensor(m.x, device="cuda")
    v = torch.tensor(np.random.default_rng(3).standard_normal(m.x.shape), device="cuda")
    v[:, torch.tensor(m.fixed[0].astype(bool), device="cuda")] = 0.0
    y = ctx.hess_apply(x, v).cpu().numpy()
    node = int(np.flatnonzero(m.fixed[0] == 0)[0])
    w = v.clone()
    w[0, node] = bad
    z = ctx.hess_apply(x, w).cpu().numpy()
    hit = np.zeros(m.nnode, dtype=bool)
    for row in m.elem_nodes:
        if node in row:
            hit[row] = True
    free = m.fixed == 0
    assert np.isnan(z[free & hit[None, :]]).all()
    assert np.array_equal(z[free & ~hit[None, :]], y[free & ~hit[None, :]])


@pytest.mark.parametrize("dim,order,nq,metric", CASES)
def test_stored_product_with_values_that_are_not_finite(dim, order, nq, metric):
    """A direction that is not finite at one node spoils that node's elements
    only."""
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = _mesh(dim, order, nq, metric)
    ctx = tm.Context.from_mesh(m)
    ctx.set_deterministic(True)
    x = torch.tensor(m.x, device="cuda")
    v = torch.tensor(np.random.default_rng(3).standard_normal(m.x.shape), device="cuda")
    ctx.linearize(x)
    y = ctx.hess_apply_pa(v).cpu().numpy()
    node = int(np.flatnonzero(m.fixed[0] == 0)[0])
    hit = np.zeros(m.nnode, dtype=bool)
    for row in m.elem_nodes:
        if node in row:
            hit[row] = True
    free = m.fixed == 0
    w = v.clone()
    w[:, node] = float("nan")   # (every component: a stored Hessian need not mix them)
    z = ctx.hess_apply_pa(w).cpu().numpy()
    assert np.isnan(z[free & hit[None, :]]).all()
    assert np.array_equal(z[free & ~hit[None, :]], y[free & ~hit[None, :]])
