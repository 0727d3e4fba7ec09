"""The ends of the exponent range in the FP64 fixed-point kernels: results that
underflow become zero (nothing is represented below about 2^-1010), and
results that are zero but for rounding are no larger than it."""
import numpy as np
import pytest

from paper_1807_09807_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu

CASES = [(3, 1, 3, 303), (3, 2, 4, 302), (3, 3, 5, 303), (3, 4, 6, 303)]


def _mesh(dim, order, nq, metric, jit=0.08):
    nx = (3, 2, 2)[:dim]
    x, en, fx = mg.structured(dim, order, nx)
    x = np.ascontiguousarray(mg.jitter(x, fx, jit / (order * 3), 5))
    return mg.Mesh(dim=dim, order=order, nx=nx, x=x, x_ideal=x, elem_nodes=en, fixed=fx, nq=nq, quad_kind=mg.GL,
                   metric=metric)


@pytest.mark.parametrize("dim,order,nq,metric", CASES)
def test_stored_product_of_directions_of_any_exponent(dim, order, nq, metric):
    """A direction times a power of two: the same digits. Where the product
    nears the end of the range its sums lose their last bits to the common
    exponent: an error of at most 2^-1000 of an entry of H, the largest of
    which is below 2^10 here."""
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = _mesh(dim, order, nq, metric)
    ctx = tm.Context.from_mesh(m)
    ctx.set_deterministic(True)
    x = torch.tensor(m.x, device="cuda")
    v = torch.tensor(np.random.default_rng(2).standard_normal(m.x.shape), device="cuda")
    ctx.linearize(x)
    y = ctx.hess_apply_pa(v)
    for k in (-600, -40, 40, 600):
        assert torch.equal(ctx.hess_apply_pa(v * 2.0 ** k), y * 2.0 ** k)
    for k in (-920, -960, -990, -1000, -1010):
        z = ctx.hess_apply_pa(v * 2.0 ** k)
        assert z.isfinite().all() and (z - y * 2.0 ** k).abs().max() <= 2.0 ** -990
    assert not ctx.hess_apply_pa(torch.zeros_like(v)).any()
    assert not ctx.hess_apply_pa(torch.zeros_like(v) * v.sign()).any()   # zeros of both signs
    assert not ctx.hess_apply(x, torch.zeros_like(v) * v.sign()).any()


@pytest.mark.parametrize("order,nq", [(1, 2), (2, 3), (2, 4), (3, 4), (3, 5), (4, 6)])
def test_gradient_of_the_ideal_mesh(order, nq):
    """Unit cubes: P = 0 but for rounding, some eps times its terms (each of
    order 1 here, times the derivative tables' entries, below 64)."""
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    x, en, fx = mg.structured(3, order, (2, 2, 2))
    x = np.ascontiguousarray(2.0 * x)
    fx = np.zeros_like(fx)
    ctx = tm.Context(3, order, x.shape[1], None, fx, nq, 303, structured=[2, 2, 2], nelem=8)
    xd = torch.tensor(x, device="cuda")
    tol = 64 * 64 * 2.2e-16
    assert ctx.gradient(xd).abs().max() <= tol
    assert ctx.energy_gradient(xd)[0].abs().max() <= tol
    g, y = ctx.gradient_hess_apply(xd, xd)   # (x itself: dP[T] = -P)
    assert g.abs().max() <= tol and y.abs().max() <= tol
    assert ctx.hess_apply(xd, xd).abs().max() <= tol
    ctx.linearize(xd)
    assert ctx.hess_apply_pa(xd).abs().max() <= tol
