"""The FP64 kernels' fixed-point numbers have one exponent where fields differ in
size: a direction whose components differ by powers of ten shares one on the
mu303 path, a stored Hessian's entries share them by rows, and elements can be
long and short in reference directions. Against the same formulas in extended
precision, component by component: the error is that of plain FP64 (up to four
times the oracle's largest, which FP64 sums in another order reach too, or 20
eps where the oracle's happens to be small)."""
import numpy as np
import pytest

import oracle
from paper_1807_09807_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu

L = np.longdouble


def cof(a, b):
    """Bilinear form of the cofactor matrix: cof(a, a) = cof a."""
    c = np.zeros_like(a)
    for i in range(3):
        for j in range(3):
            r1, r2, c1, c2 = (i + 1) % 3, (i + 2) % 3, (j + 1) % 3, (j + 2) % 3
            c[:, i, j] = (a[:, r1, c1] * b[:, r2, c2] - a[:, r1, c2] * b[:, r2, c1] + b[:, r1, c1] * a[:, r2, c2] -
                          b[:, r1, c2] * a[:, r2, c1]) / 2
    return c


def exact(orc, en, x, v):
    """Gradient and Hessian action of mu303 = |T|^2 / (3 tau^(2/3)) - 1, W = I."""
    w, gp = (t.astype(L) for t in orc.tables())
    g, y = np.zeros(x.shape, L), np.zeros(x.shape, L)
    for e in en:
        T, V = np.einsum("qnd,an->qad", gp, x[:, e].astype(L)), np.einsum("qnd,an->qad", gp, v[:, e].astype(L))
        C, D = cof(T, T), 2 * cof(T, V)
        tau, I1 = (T[:, 0] * C[:, 0]).sum(1), (T * T).sum((1, 2))
        t, d = (T * V).sum((1, 2)), (C * V).sum((1, 2))
        cA = L(2) / 3 * tau ** (-L(2) / 3)
        ct = -I1 / 3 / tau * cA
        dcA = -L(2) / 3 * cA / tau * d
        dct = (-L(2) / 3 * t + I1 / 3 / tau * d) / tau * cA - I1 / 3 / tau * dcA
        f = [s[:, None, None] for s in (cA, ct, dcA, dct)]
        g[:, e] += np.einsum("q,qab,qnb->an", w, f[0] * T + f[1] * C, gp)
        y[:, e] += np.einsum("q,qab,qnb->an", w, f[0] * V + f[2] * T + f[3] * C + f[1] * D, gp)
    return g, y


def errors(a, ref):
    return np.linalg.norm((a - ref).astype(float), axis=1) / np.linalg.norm(ref.astype(float), axis=1)


def check(order, nq, nx, x, v):
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    en, fx = mg.structured(3, order, nx)[1:]
    fx = np.zeros_like(fx)
    x, v = np.ascontiguousarray(x), np.ascontiguousarray(v)
    orc = oracle.Problem(3, order, en, x.shape[1], fx, nq, 303)
    ctx = tm.Context(3, order, x.shape[1], None, fx, nq, 303, structured=list(nx), nelem=len(en))
    xd, vd = torch.tensor(x, device="cuda"), torch.tensor(v, device="cuda")
    assert ctx.energy(xd)[0] == tm.OK
    g, y = exact(orc, en, x, v)
    eg, ey = errors(orc.gradient(x), g), errors(orc.hess_apply(x, v), y)
    ctx.linearize(xd)
    for name, out, ref, e in [("gradient", ctx.gradient(xd), g, eg), ("action", ctx.hess_apply(xd, vd), y, ey),
                              ("both, g", ctx.gradient_hess_apply(xd, vd)[0], g, eg),
                              ("both, y", ctx.gradient_hess_apply(xd, vd)[1], y, ey),
                              ("stored", ctx.hess_apply_pa(vd), y, ey)]:
        got = errors(out.cpu().numpy(), ref)
        assert got.max() <= max(4 * e.max(), 20 * 2.2e-16), (name, got, e)


@pytest.mark.parametrize("order,nq", [(1, 2), (2, 4), (3, 5)])
@pytest.mark.parametrize("sizes", [(1, 1e-8, 1e-8), (1e-8, 1, 1e-4), (1, 1, 1e-12), (0, 1, 0)])
def test_directions_with_components_of_different_size(order, nq, sizes):
    x, en, fx = mg.structured(3, order, (2, 2, 2))
    x = mg.jitter(x, fx, 0.08 / (order * 2), 5)
    v = np.random.default_rng(1).standard_normal(x.shape) * np.array(sizes, dtype=float)[:, None]
    check(order, nq, (2, 2, 2), x, v)


@pytest.mark.parametrize("order,nq", [(2, 4), (3, 5)])
@pytest.mark.parametrize("aspect", [30, 1000])
@pytest.mark.parametrize("turned", [False, True])   # long in a row of A, or in a reference direction of turned elements
@pytest.mark.parametrize("direction", ["random", "along", "linear"])
def test_long_elements(order, nq, aspect, turned, direction):
    rng = np.random.default_rng(0)
    X = mg.structured(3, order, (1, 1, 1))[0]
    X = X + 0.02 / order * rng.standard_normal(X.shape)
    S = np.diag([aspect, 1.0, 1.0])
    Q = np.linalg.qr(rng.standard_normal((3, 3)))[0] if turned else np.eye(3)
    v = {"random": rng.standard_normal(X.shape), "along": np.stack([np.sin(2 * X[0]), X[0] ** 2, np.cos(X[0])]),
         "linear": Q @ S @ np.stack([X[0] * X[1], X[1] * X[2], X[2] * X[0]])}[direction]
    check(order, nq, (1, 1, 1), Q @ S @ X * (1 if np.linalg.det(Q) > 0 else np.array([[-1.0], [1.0], [1.0]])), v)
