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


@pytest.mark.parametrize("order,nq", [(1, 2), (2, 4), (3, 5), (4, 6)])
@pytest.mark.parametrize("k", [-330, -250, -150, -100, -43, -42, -41, -38, -37, 37, 38, 41, 42, 43, 100, 150, 250, 330])
def test_meshes_of_any_size(order, nq, k):
    """x times 2^k, both sides of the sizes the fixed-point stage of mu303 takes:
    mu is scale invariant, so F stays, det A takes 2^(3k), the gradient 2^-k and
    the Hessian action 2^-2k. (The Hessian's tau^(-8/3) |T|^2 leaves the FP64
    range by itself above |k| = 160.) 1e-11, as between two ways to compute it."""
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = _mesh(3, order, nq, 303)
    ctx = tm.Context.from_mesh(m)
    ctx.set_deterministic(True)
    x = torch.tensor(m.x, device="cuda")
    v = torch.tensor(np.random.default_rng(2).standard_normal(m.x.shape), device="cuda")
    s = 2.0 ** k
    F, g, y = ctx.energy(x), ctx.gradient(x), ctx.hess_apply(x, v)

    def near(a, b):
        return bool((a - b).norm() <= 1e-11 * b.norm())

    Fs = ctx.energy(x * s)
    assert Fs[0] == F[0] and abs(Fs[1] - F[1]) <= 1e-11 * F[1] and abs(Fs[2] / s / s / s - F[2]) <= 1e-11 * F[2]
    assert near(ctx.gradient(x * s) * s, g)
    ge, Fe, md = ctx.energy_gradient(x * s)
    assert near(ge * s, g) and abs(Fe.item() - F[1]) <= 1e-11 * F[1] and md.item() == Fs[2]
    if abs(k) > 150:
        return
    assert near(ctx.hess_apply(x * s, v) * s * s, y)
    gh, yh = ctx.gradient_hess_apply(x * s, v)
    assert near(gh * s, g) and near(yh * s * s, y)
    ctx.linearize(x * s)
    assert near(ctx.hess_apply_pa(v) * s * s, y)


@pytest.mark.parametrize("order,nq", [(1, 2), (2, 4), (3, 5), (4, 6)])
@pytest.mark.parametrize("kx", [-39, 0, 39])
@pytest.mark.parametrize("kv", [-880, -616, -606, 602, 612, 850])
def test_directions_of_any_size(order, nq, kx, kv):
    """v times 2^kv at sizes of x near the ends of that range, on both sides of
    the sizes of v the stage takes. (The terms of dP go as |v| |x|^-4.)"""
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = _mesh(3, order, nq, 303)
    ctx = tm.Context.from_mesh(m)
    ctx.set_deterministic(True)
    x = torch.tensor(m.x, device="cuda")
    v = torch.tensor(np.random.default_rng(2).standard_normal(m.x.shape), device="cuda")
    y = ctx.hess_apply(x, v)
    z = ctx.hess_apply(x * 2.0 ** kx, v * 2.0 ** kv) * 2.0 ** -kv * 2.0 ** (2 * kx)
    assert (z - y).norm() <= 1e-11 * y.norm()


@pytest.mark.parametrize("order,nq,metric", [(1, 2, 303), (2, 4, 302), (3, 5, 303), (3, 4, 98)])
@pytest.mark.parametrize("target", ["unit", "scaled"])   # closed forms, nine directions
def test_stored_product_of_a_mesh_with_inverted_points(order, nq, metric, target):
    """Points with det T <= 0 have no Hessian: zeros, packed with the others'.
    The recomputed action skips them; 1e-10 of the largest value, as the points
    beside them have det T small."""
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = _mesh(3, order, nq, metric)
    n = int(np.flatnonzero(m.fixed[0] == 0)[0])
    m.x[0, n] += 2.0
    ctx = tm.Context.from_mesh(m, target_scale=0.5 if target == "scaled" else None)
    x = torch.tensor(m.x, device="cuda")
    assert ctx.energy(x)[0] != tm.OK
    v = torch.tensor(np.random.default_rng(2).standard_normal(m.x.shape), device="cuda")
    ctx.linearize(x)
    y, z = ctx.hess_apply_pa(v), ctx.hess_apply(x, v)
    assert z.isfinite().all() and (y - z).abs().max() <= 1e-10 * z.abs().max()
