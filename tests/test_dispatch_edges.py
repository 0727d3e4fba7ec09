"""Sizes and forms at which the FP64 element kernels and the MINRES vector
kernels change: half a warp per 2D element from 1216 elements on, the
fixed-point pointwise stage of mu303 against the general one, the closed-form
second derivatives of mu302 and mu98, the one-cluster MINRES up to 2048 and
8192 unknowns, the scalar step in its own kernel above 150000."""
import numpy as np
import pytest

import oracle
from paper_1807_09807_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu


def _mesh(dim, order, nx, nq, metric, jit=0.08, kind=mg.GL):
    x, en, fx = mg.structured(dim, order, nx)
    x = np.ascontiguousarray(mg.jitter(x, fx, jit / (order * max(nx)), 5))
    return mg.Mesh(dim=dim, order=order, nx=nx, x=x, x_ideal=x, elem_nodes=en, fixed=fx, nq=nq, quad_kind=kind,
                   metric=metric)


def _oracle(m, **kw):
    return oracle.Problem(m.dim, m.order, m.elem_nodes, m.nnode, m.fixed, m.nq, m.metric, quad_kind=m.quad_kind, **kw)


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("nx", [(27, 45), (32, 38), (35, 35)])   # 1215, 1216 and an odd number above
@pytest.mark.parametrize("order,nq,structured", [(1, 2, True), (2, 3, False), (2, 5, True), (3, 5, False), (4, 6, True)])
def test_half_a_warp_per_element(nx, order, nq, structured):
    """1e-11 as for the 3D elements: W = I makes T of order 1 / 35, and the
    oracle's own sums differ by some 1e-13 from another order."""
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = _mesh(2, order, nx, nq, 2)
    ctx, orc = tm.Context.from_mesh(m, structured=structured), _oracle(m)
    x, v = torch.tensor(m.x, device="cuda"), np.random.default_rng(1).standard_normal(m.x.shape)
    vd = torch.tensor(v, device="cuda")
    F, Fo = ctx.energy(x), orc.energy(m.x)
    assert abs(F[1] - Fo[1]) <= 1e-11 * abs(Fo[1]) and abs(F[2] - Fo[2]) <= 1e-11 * abs(Fo[2])
    go, yo = orc.gradient(m.x), orc.hess_apply(m.x, v)
    g, F2, md = ctx.energy_gradient(x)
    assert md.item() == F[2] and abs(F2.item() - F[1]) <= 1e-13 * abs(F[1])
    assert _rel(g.cpu().numpy(), go) <= 1e-11 and _rel(ctx.gradient(x).cpu().numpy(), go) <= 1e-11
    assert _rel(ctx.hess_apply(x, vd).cpu().numpy(), yo) <= 1e-11
    g, y = ctx.gradient_hess_apply(x, vd)
    assert _rel(g.cpu().numpy(), go) <= 1e-11 and _rel(y.cpu().numpy(), yo) <= 1e-11
    ctx.linearize(x)
    assert _rel(ctx.hess_apply_pa(vd).cpu().numpy(), yo) <= 1e-11


@pytest.mark.parametrize("order,nq,kind", [(1, 2, mg.GL), (1, 3, mg.GL), (2, 3, mg.GL), (2, 4, mg.GL),
                                           (3, 4, mg.GL), (3, 5, mg.GL), (4, 5, mg.GL), (4, 6, mg.GL)])
@pytest.mark.parametrize("structured,stretch", [(True, 1.0), (False, 1.0), (True, 64.0)])
def test_mu303_with_unit_targets_against_the_general_path(order, nq, kind, structured, stretch):
    """W = I given as the scaled target 1.0 takes the FP64 pointwise stage. A
    stretched axis makes the components' exponents differ by more than the
    fixed-point stage takes (then both are the general path). P cancels to
    some 1e-2 of its terms here: 1e-11 as above; F to as many digits less."""
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = _mesh(3, order, (3, 2, 2), nq, 303, kind=kind)
    m.x = np.ascontiguousarray(m.x * np.array([1.0, stretch, 1.0])[:, None])
    a = tm.Context.from_mesh(m, structured=structured)
    b = tm.Context.from_mesh(m, structured=structured, target_scale=1.0)
    for c in (a, b):
        c.set_deterministic(True)
    x = torch.tensor(m.x, device="cuda")
    v = torch.tensor(np.random.default_rng(1).standard_normal(m.x.shape), device="cuda")
    Fa, Fb = a.energy(x), b.energy(x)
    assert Fa[0] == Fb[0] and abs(Fa[1] - Fb[1]) <= 1e-11 * abs(Fb[1]) and abs(Fa[2] - Fb[2]) <= 1e-11 * abs(Fb[2])
    ga, gb = a.gradient(x).cpu().numpy(), b.gradient(x).cpu().numpy()
    ya, yb = a.hess_apply(x, v).cpu().numpy(), b.hess_apply(x, v).cpu().numpy()
    assert _rel(ga, gb) <= 1e-11 and _rel(ya, yb) <= 1e-11
    g, y = a.gradient_hess_apply(x, v)
    assert _rel(g.cpu().numpy(), gb) <= 1e-11 and _rel(y.cpu().numpy(), yb) <= 1e-11
    g, F2, md = a.energy_gradient(x)
    assert _rel(g.cpu().numpy(), gb) <= 1e-11 and md.item() == Fa[2] and abs(F2.item() - Fa[1]) <= 1e-13 * abs(Fa[1])
    # an inverted element: both see it
    n = int(np.flatnonzero(m.fixed[0] == 0)[0])
    m.x[0, n] += 2.0
    x = torch.tensor(m.x, device="cuda")
    Fa, Fb = a.energy(x), b.energy(x)
    assert Fa[0] == Fb[0] != tm.OK and Fa[2] < 0 and abs(Fa[2] - Fb[2]) <= 1e-11 * abs(Fb[2])


@pytest.mark.parametrize("dim,order,nq,metric", [(2, 2, 3, 98), (2, 3, 5, 98), (3, 1, 2, 302), (3, 2, 4, 302), (3, 2, 3, 98),
                                                 (3, 3, 5, 302), (3, 3, 5, 98)])
@pytest.mark.parametrize("target", ["unit", "scaled", "constant", "per_point", "second"])
@pytest.mark.parametrize("precision,tol", [("fp64", 1e-11), ("fp32", 1e-5)])
def test_second_derivatives_of_mu302_and_mu98(dim, order, nq, metric, target, precision, tol):
    """Recomputed, with the gradient and stored, for every kind of target (tol:
    the FP32 form's is that of its other products)."""
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = _mesh(dim, order, (3, 2, 2)[:dim], nq, metric)
    rng = np.random.default_rng(7)
    kw, okw = {}, {}
    if target == "scaled":
        kw, okw = dict(target_scale=0.25), dict(wkind=oracle.W_CONST, W=0.25 * np.eye(dim))
    if target == "constant":
        m.W = 0.3 * (np.eye(dim) + 0.1 * rng.standard_normal((dim, dim)))
        okw = dict(wkind=oracle.W_CONST, W=m.W)
    if target == "per_point":
        W = 0.3 * (np.eye(dim) + 0.1 * rng.standard_normal((m.nelem, m.Q, dim, dim)))
        kw, okw = dict(W_per_qp=W), dict(wkind=oracle.W_PER_QP, W=W)
    ctx = tm.Context.from_mesh(m, precision=tm.FP64 if precision == "fp64" else tm.FP32_MIXED, **kw)
    if target == "second":   # the metric as the second term
        first = 2 if dim == 2 else 303
        ctx = tm.Context.from_mesh(m, metric=first, precision=tm.FP64 if precision == "fp64" else tm.FP32_MIXED)
        ctx.set_composite(metric, 0.3 * np.eye(dim))
        okw = dict(metric2=metric, W2=0.3 * np.eye(dim))
        m.metric = first
    orc = _oracle(m, **okw)
    x, v = torch.tensor(m.x, device="cuda"), rng.standard_normal(m.x.shape)
    vd = torch.tensor(v, device="cuda")
    go, yo = orc.gradient(m.x), orc.hess_apply(m.x, v)
    assert _rel(ctx.hess_apply(x, vd).cpu().numpy(), yo) <= tol
    g, y = ctx.gradient_hess_apply(x, vd)
    assert _rel(g.cpu().numpy(), go) <= tol * 10 and _rel(y.cpu().numpy(), yo) <= tol
    ctx.linearize(x)
    assert _rel(ctx.hess_apply_pa(vd).cpu().numpy(), yo) <= tol


@pytest.mark.parametrize("nx,unknowns", [((2, 2), 18), ((31, 31), 2048), ((40, 24), 2050), ((63, 63), 8192), ((40, 99), 8200),
                                         ((273, 273), 150152)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_minres_vectors_in_one_cluster(nx, unknowns, precision):
    """After twelve iterations the oracle's iterate (rounding grows little in
    so few: 1e-10, and the FP32 form's operator and vectors 1e-4), and solved,
    the residual asked for (FP32: of its own operator, as far as its vectors
    carry)."""
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    m = _mesh(2, 1, nx, 2, 2)
    assert m.x.size == unknowns
    orc = _oracle(m)
    ctx = tm.Context.from_mesh(m, precision=tm.FP64 if precision == "fp64" else tm.FP32_MIXED)
    x = torch.tensor(m.x, device="cuda")
    b = np.random.default_rng(3).standard_normal(m.x.shape) * (1 - m.fixed)
    bd = torch.tensor(b, device="cuda")
    fp64 = precision == "fp64"
    if unknowns > 18:   # (18: two free unknowns, solved in two iterations)
        p, _ = ctx.krylov_solve(x, bd, krylov_rtol=1e-14, krylov_maxit=12)
        po, _ = orc.minres(m.x, b, rtol=1e-14, maxit=12)
        assert _rel(p.cpu().numpy(), po) <= (1e-10 if fp64 else 1e-4)
    if unknowns > 100000:
        return
    p, it = ctx.krylov_solve(x, bd, krylov_rtol=1e-9 if fp64 else 1e-5, krylov_maxit=5000)
    assert it > 0
    assert _rel(orc.hess_apply(m.x, p.cpu().numpy()), b) <= (1e-8 if fp64 else 1e-4 * 10)
