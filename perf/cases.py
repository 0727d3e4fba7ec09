"""The work that users of this library have it do, as cases that can be timed.

Every case goes through the public entry points: `tmop.Context` (objective,
gradient, Hessian actions, Krylov and Newton solves), `autograd.tmop_energy`
and the proposal network of `learned`. A case is a dict of plain values;
"op" says which call it makes:

  step      gradient and Hessian action at the same x (the benchmark step)
  trial     objective, min det A and gradient of one line-search trial
  hess      one matrix-free Hessian action
  products  one linearisation and a few stored-Hessian products with it
  krylov    MINRES on H p = g for a fixed number of iterations
  newton    a whole Newton solve from a perturbed mesh
  autograd  the objective as a torch function, and its backward
  mlp       loss and gradients of the proposal network on one minibatch
  proposal  patch features, network, displaced mesh and its objective

Meshes are grids of order-k quads or hexes on the unit square or cube with
every interior node moved at random by a share of the node spacing, boundary
nodes fixed, as the library's own workloads are.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1807_09807_gb300 import autograd as tag
from paper_1807_09807_gb300 import learned
from paper_1807_09807_gb300 import meshgen as mg
from paper_1807_09807_gb300 import tmop as tm

PRECISION = {"fp64": tm.FP64, "mixed": tm.FP32_MIXED, "bulk": tm.FP32_BULK}
PAIRS = {2: {1: (2, 3), 2: (3, 4, 5), 3: (4, 5, 6), 4: (5, 6)}, 3: {1: (2, 3), 2: (3, 4), 3: (4, 5), 4: (5, 6)}}


def _mesh_case(name, op, dim, order, n, nq, metric, precision="fp64", **more):
    c = dict(name=name, op=op, dim=dim, order=order, nx=n[0], ny=n[1], nz=n[2] if dim == 3 else 1, nq=nq,
             metric=metric, precision=precision, target="identity", deform="none", jitter=0.1, structured=True,
             deterministic=False)
    c.update(more)
    return c


def listed():
    return [
        # the library's headline workload: 9.1 M unknowns, one gradient and one
        # Hessian action at the same positions
        _mesh_case("step_hex3_48", "step", 3, 3, (48, 48, 48), 5, 303, deform="shear"),
        # what the Newton line search evaluates at every trial, on the order-2 mesh
        _mesh_case("trial_hex2_32", "trial", 3, 2, (32, 32, 32), 4, 303, deform="shear"),
        # an inner solve in FP64: linearisation, then MINRES iterations on a
        # mid-size mesh with ragged sides
        _mesh_case("krylov_hex3_24", "krylov", 3, 3, (24, 21, 17), 5, 303, deform="shear", iters=24),
        # the time to a converged mesh of the headline workload, in the form a
        # user in a hurry takes: FP32 Hessian, two-level preconditioner
        _mesh_case("newton_mixed_hex3_48", "newton", 3, 3, (48, 48, 48), 5, 303, "mixed", deform="shear", precond=2),
        # a whole 2D solve in FP64 with the two-level preconditioner
        _mesh_case("newton_quad3_64", "newton", 2, 3, (64, 64), 5, 2, deform="sine", precond=2),
        # the smallest solve: 289 nodes, plain MINRES, bound by launches and latency
        _mesh_case("newton_quad2_8", "newton", 2, 2, (8, 8), 4, 2, jitter=0.15, precond=0),
        # the smallest call: the objective in a torch program, with its backward
        _mesh_case("autograd_quad2_8", "autograd", 2, 2, (8, 8), 4, 2, jitter=0.15),
        # the FP32 Hessian action recomputed from x (memory-lean Krylov operator)
        _mesh_case("hess_mixed_hex3_48", "hess", 3, 3, (48, 48, 48), 5, 303, "mixed", deform="shear"),
        # the FP32 Krylov operator: one linearisation and its products, ragged sides
        _mesh_case("products_mixed_hex3_40", "products", 3, 3, (40, 37, 43), 5, 303, "mixed", deform="shear", count=8),
        # unstructured connectivity, order 4, size-preserving per-point targets
        _mesh_case("step_quad4_local", "step", 2, 4, (150, 117), 6, 7, target="local", structured=False),
        # one training minibatch of the proposal network
        dict(name="mlp_4096", op="mlp", order=3, hidden=256, batch=4096),
        # the proposal on a mesh that is to be solved
        _mesh_case("proposal_quad3_128", "proposal", 2, 3, (128, 128), 5, 2, jitter=0.15, hidden=256),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["step", "step", "trial", "hess", "products", "krylov", "newton", "autograd", "mlp", "proposal"])
    if op == "mlp":
        return dict(op="mlp", order=rng.choice([2, 3, 4]), hidden=64 * rng.randint(1, 4),
                    batch=64 * _log_int(rng, 1, 64))
    dim = 2 if op == "proposal" else rng.choice([2, 3, 3])
    order = rng.randint(2, 3) if op in ("newton", "proposal") else rng.randint(1, 4)
    nq = rng.choice([q for q in PAIRS[dim][order] if q > order])
    # unknowns spread over the range of the listed cases
    top = {"krylov": 1.2e6, "newton": 6e4}.get(op, 6e6)
    side = math.exp(rng.uniform(math.log(3 * order), math.log((top / dim) ** (1.0 / dim)))) / order
    n = [max(3, int(round(side * rng.uniform(0.75, 1.25)))) for _ in range(dim)]
    c = _mesh_case("", op, dim, order, n, nq, rng.choice((2, 7, 9, 77, 98) if dim == 2 else (303, 303, 302, 98)))
    del c["name"]
    c["precision"] = rng.choice(["fp64", "fp64", "mixed"] + (["bulk"] if op in ("step", "trial", "hess") else []))
    c["jitter"] = round(rng.uniform(0.05, 0.12), 3)
    c["deform"] = rng.choice(["none", "sine"]) if dim == 2 else rng.choice(["none", "shear"])
    if c["metric"] in (7, 9, 77, 98):   # size matters: a target of the elements' size
        c["target"] = rng.choice(["scaled", "local"])
    if op in ("newton", "proposal", "krylov"):
        c.update(metric=2 if dim == 2 else 303, target="identity")
    if op in ("step", "trial", "hess", "products"):
        c["structured"] = rng.random() < 0.75
        c["deterministic"] = rng.random() < 0.15
    if op == "newton":
        c.update(precond=2, deform="none")
    if op == "krylov":
        c["iters"] = 6 * rng.randint(2, 4)
    if op == "products":
        c["count"] = rng.randint(4, 12)
    if op == "proposal":
        c["hidden"] = 256
        c["ny"] = c["nx"] = max(c["nx"], 8)
        c.update(deform="none", precision="fp64")
    return c


# ------------------------------------------------------------------ inputs
def _sizes(c):
    return [c["nx"], c["ny"], c["nz"]][: c["dim"]]


def _lattice(c):
    """Undisturbed positions [d][nnode] (before the shear) and the fixed-dof mask, on the GPU."""
    ax = [torch.tensor(mg.lattice_coordinates(c["order"], n), device="cuda") for n in _sizes(c)]
    g = torch.meshgrid(*reversed(ax), indexing="ij")
    x = torch.stack([t.reshape(-1) for t in reversed(g)])
    bnd = torch.zeros(g[0].shape, dtype=torch.bool, device="cuda")
    for d in range(c["dim"]):
        bnd.select(d, 0).fill_(True)
        bnd.select(d, -1).fill_(True)
    return x, bnd.reshape(1, -1).expand(c["dim"], -1).contiguous()


def _elem_nodes(c):
    """Node ids [nelem][(k+1)^d] of a lexicographic grid, on the GPU."""
    k, n = c["order"], c["order"] + 1
    s = _sizes(c)
    per = [k * v + 1 for v in s]
    first = torch.zeros(1, dtype=torch.int64, device="cuda")
    local = torch.zeros(1, dtype=torch.int64, device="cuda")
    stride = 1
    for d in range(c["dim"]):   # x fastest
        first = (torch.arange(s[d], device="cuda") * (k * stride))[:, None] + first[None, :]
        local = (torch.arange(n, device="cuda") * stride)[:, None] + local[None, :]
        first, local = first.reshape(-1), local.reshape(-1)
        stride *= per[d]
    return first[:, None] + local[None, :]


def _positions(c, seed):
    x, fixed = _lattice(c)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    if c["deform"] == "sine":
        x[0] += 0.05 * torch.sin(2 * math.pi * x[0]) * torch.sin(2 * math.pi * x[1])
    h = 1.0 / (c["order"] * max(_sizes(c)))
    u = torch.rand(x.shape, dtype=torch.float64, device="cuda", generator=gen) * 2 - 1
    x = x + c["jitter"] * h * u * (~fixed)
    if c["deform"] == "shear":
        X, Y, Z = x
        x = torch.stack([X + 0.2 * Y + 0.1 * Y * Z, Y + 0.1 * Z, Z])
    return x.contiguous(), fixed, gen


def _scale(c):
    """Edge length of a cube of the mean element size (all grids here fill a unit volume)."""
    return float(np.prod(_sizes(c))) ** (-1.0 / c["dim"])


def prepare(case, seed):
    c = dict(case)
    if c["op"] == "mlp":
        gen = torch.Generator(device="cuda").manual_seed(seed)
        n_in, n_out = learned.n_features(c["order"]), learned.n_targets(c["order"])
        net = learned.MLP(n_in, n_out, c["hidden"], seed=seed % 1000)
        X = torch.zeros((c["batch"], net.ld), dtype=torch.bfloat16, device="cuda")
        X[:, :n_in] = 0.1 * torch.randn((c["batch"], n_in), device="cuda", generator=gen)
        T = 0.05 * torch.randn((c["batch"], n_out), device="cuda", generator=gen)
        loss = torch.zeros((), dtype=torch.float64, device="cuda")
        return dict(c, net=net, X=X.view(torch.int16), T=T, loss=loss)
    x, fixed, gen = _positions(c, seed)
    fx = fixed.to(torch.uint8).cpu().numpy()
    en = None if c["structured"] else _elem_nodes(c).to(torch.int32).cpu().numpy()
    kind, scale = (tm.W_SCALED, _scale(c)) if c["target"] == "scaled" else (tm.W_IDENTITY, 1.0)
    ctx = tm.Context(c["dim"], c["order"], x.shape[1], en, fx, c["nq"], c["metric"],
                     structured=_sizes(c) if c["structured"] else None, target_kind=kind, target_scale=scale,
                     precision=PRECISION[c["precision"]], nelem=int(np.prod(_sizes(c))))
    if c["target"] == "local":   # each element keeps the size it has before the jitter
        ctx.set_targets_from_positions(tm.WT_LOCAL_SIZE, _positions(dict(c, jitter=0.0), 0)[0])
    if c["deterministic"]:
        ctx.set_deterministic(True)
    st = dict(c, ctx=ctx, x=x)
    if c["op"] in ("step", "hess"):
        st["v"] = torch.randn(x.shape, dtype=torch.float64, device="cuda", generator=gen)
    if c["op"] == "products":
        st["vs"] = [torch.randn(x.shape, dtype=torch.float64, device="cuda", generator=gen) for _ in range(c["count"])]
    if c["op"] == "krylov":
        st["b"] = ctx.gradient(x)
    if c["op"] == "proposal":
        net = learned.MLP(learned.n_features(c["order"]), learned.n_targets(c["order"]), c["hidden"], seed=seed % 1000)
        host = mg.Mesh(dim=2, order=c["order"], nx=(c["nx"], c["ny"]), x=np.empty((2, x.shape[1])), x_ideal=None,
                       elem_nodes=np.empty((c["nx"] * c["ny"], 0), dtype=np.int32), fixed=fx, nq=c["nq"],
                       metric=c["metric"])
        st.update(net=net, mesh=host, fixed=fixed.to(torch.uint8))
    return st


# ------------------------------------------------------------------ one pass
def run(st):
    op = st["op"]
    if op == "mlp":
        st["net"].gradients(st["X"], st["T"], st["loss"])
        return {"loss": st["loss"], "gradients": st["net"].get(1)}
    ctx, x = st["ctx"], st["x"]
    if op == "step":
        return ctx.gradient_hess_apply(x, st["v"])
    if op == "trial":
        g, F, min_det = ctx.energy_gradient(x)
        return {"g": g, "F": F, "min_det": min_det}
    if op == "hess":
        return ctx.hess_apply(x, st["v"])
    if op == "products":
        ctx.linearize(x)
        return [ctx.hess_apply_pa(v) for v in st["vs"]]
    if op == "krylov":
        return ctx.krylov_solve(x, st["b"], krylov_rtol=1e-14, krylov_maxit=st["iters"])[0]
    if op == "newton":
        y = x.clone()
        r = ctx.newton_solve(y, max_newton=30, precond=st["precond"])
        return {"x": y, "min_det": r.report["min_detA"], "status": r.status}
    if op == "autograd":
        y = x.detach().requires_grad_(True)
        F = tag.tmop_energy(y, ctx)
        F.backward()
        return {"F": F.detach(), "g": y.grad}
    if op == "proposal":
        m, net = st["mesh"], st["net"]
        rows = (m.nelem + 63) // 64 * 64
        X = torch.zeros((rows, net.ld), dtype=torch.int16, device=x.device)
        learned.features(m, x, net.ld, out=X[: m.nelem])
        Y = net.forward(X)[: m.nelem].contiguous()
        xp = learned.apply(m, x, st["fixed"], Y)
        status, F, min_det = ctx.energy(xp)
        return {"features": X, "x": xp, "F": F, "min_det": min_det, "Y": Y[:, : net.n_out], "status": status}
    raise ValueError(op)


# ------------------------------------------------------------------ what a pass cannot do without
def _map_fmas(c):
    """Multiply-adds of one forward and of one adjoint sum-factorised contraction of an element."""
    n, q = c["order"] + 1, c["nq"]
    if c["dim"] == 2:
        return 2 * (n * q * 2 * n + q * q * 2 * n), 2 * (n * q * 2 * q + n * n * 2 * q)
    return (3 * (n * n * q * 2 * n + n * q * q * 3 * n + q ** 3 * 3 * n),
            3 * (n * q * q * 3 * q + n * n * q * 3 * q + n ** 3 * 2 * q))


def work(case):
    c = case
    if c["op"] == "mlp":
        h, i, o = c["hidden"], learned.n_features(c["order"]), learned.n_targets(c["order"])
        w = h * i + h * h + o * h
        # forward, and in the backward the weight gradients and all but the first layer's input gradient
        return {"bytes": c["batch"] * (2 * i + 4 * o) + 8 * w, "flops": 2 * c["batch"] * (3 * w - h * i)}
    s = _sizes(c)
    ne, Q = int(np.prod(s)), c["nq"] ** c["dim"]
    ndof = c["dim"] * int(np.prod([c["order"] * v + 1 for v in s]))
    fwd, adj = _map_fmas(c)
    point = 120 if c["dim"] == 3 else 40       # flops of P at a point; the Hessian's dP takes twice that
    grad, hess = 2 * (fwd + adj) + point * Q, 2 * (2 * fwd + adj) + 2 * point * Q
    stored = 2 * (fwd + adj) + (162 if c["dim"] == 3 else 32) * Q
    vec = 8 * ndof
    pa = ne * Q * ((14 if c["dim"] == 3 and c["metric"] in (1, 14, 303) and c["target"] != "local" else
                    c["dim"] ** 2 * (c["dim"] ** 2 + 1) // 2) * 4 if c["precision"] != "fp64" else
                   c["dim"] ** 2 * (c["dim"] ** 2 + 1) // 2 * 8)
    tgt = ne * Q * 8 * (c["dim"] ** 2 + 1) if c["target"] == "local" else 0
    if c["op"] == "step":
        return {"bytes": 4 * vec + tgt, "flops": ne * (hess + 2 * adj + point * Q // 4)}
    if c["op"] in ("trial", "autograd"):
        return {"bytes": 2 * vec + tgt, "flops": ne * grad}
    if c["op"] == "hess":
        return {"bytes": 3 * vec + tgt, "flops": ne * hess}
    if c["op"] == "products":
        return {"bytes": vec + pa + tgt + c["count"] * (pa + 2 * vec),
                "flops": ne * (2 * fwd + point * Q + c["count"] * stored)}
    if c["op"] == "krylov":
        return {"bytes": vec + pa + c["iters"] * (pa + 11 * vec),
                "flops": ne * (2 * fwd + point * Q + c["iters"] * stored) + 20 * c["iters"] * ndof}
    if c["op"] == "newton":   # five steps of 25 iterations (two-level) or 60
        its = 5 * (25 if c["precond"] == 2 else 60)
        return {"bytes": its * (pa + 11 * vec), "flops": ne * (its * stored + 6 * grad)}
    h, i, o = c["hidden"], learned.n_features(c["order"]), learned.n_targets(c["order"])
    return {"bytes": 3 * vec + ne * (2 * i + 4 * o), "flops": ne * (2 * (h * i + h * h + o * h) + 2 * fwd + point * Q)}


# ------------------------------------------------------------------ the same in 64 bits, in plain torch
def _rules(c):
    """Gauss-Legendre points and weights on [0, 1], and the Gauss-Lobatto Lagrange basis and derivative there."""
    t, w = np.polynomial.legendre.leggauss(c["nq"])
    t, w = 0.5 + 0.5 * t, 0.5 * w
    k = c["order"]
    inner = np.polynomial.legendre.Legendre.basis(k).deriv().roots()
    z = np.concatenate([[0.0], 0.5 + 0.5 * np.sort(inner.real), [1.0]])
    B, G = np.ones((len(t), k + 1)), np.zeros((len(t), k + 1))
    for i in range(k + 1):
        for j in range(k + 1):
            if j != i:
                B[:, i] *= (t - z[j]) / (z[i] - z[j])
                term = np.full(len(t), 1.0 / (z[i] - z[j]))
                for m in range(k + 1):
                    if m not in (i, j):
                        term = term * (t - z[m]) / (z[i] - z[m])
                G[:, i] += term
    dev = dict(dtype=torch.float64, device="cuda")
    return torch.tensor(B, **dev), torch.tensor(G, **dev), torch.tensor(w, **dev)


def _jacobians(c, x, en, B, G):
    """A[a][b], each [nelem, Q], of positions or displacements x [d][nnode]."""
    n, d = c["order"] + 1, c["dim"]
    A = []
    for a in range(d):
        e = x[a][en]
        e = (e - e[:, :1]).reshape([-1] + [n] * d)   # only differences matter
        row = []
        for b in range(d):
            t = e
            for axis in range(d):   # torch dimension d - axis is the coordinate `axis`
                M = G if axis == b else B
                t = torch.tensordot(t, M, dims=([d - axis], [1])).movedim(-1, d - axis)
            row.append(t.reshape(e.shape[0], -1))
        A.append(row)
    return A


def _det(T):
    if len(T) == 2:
        return T[0][0] * T[1][1] - T[0][1] * T[1][0]
    return sum(T[0][j] * (T[1][(j + 1) % 3] * T[2][(j + 2) % 3] - T[1][(j + 2) % 3] * T[2][(j + 1) % 3])
               for j in range(3))


def _mu(metric, T):
    d = len(T)
    I1, t = sum(T[a][b] ** 2 for a in range(d) for b in range(d)), _det(T)
    if metric == 2:
        return I1 / (2 * t) - 1
    if metric == 7:
        return I1 * (1 + t ** -2) - 4
    if metric == 9:
        return t * I1 + I1 / t - 4 * t
    if metric == 77:
        return 0.5 * (t - 1 / t) ** 2
    if metric == 98:
        return sum((T[a][b] - float(a == b)) ** 2 for a in range(d) for b in range(d)) / t
    if metric == 303:
        return I1 / (3 * t ** (2.0 / 3.0)) - 1
    if metric == 302:
        K = sum((T[(i + 1) % 3][(j + 1) % 3] * T[(i + 2) % 3][(j + 2) % 3] -
                 T[(i + 1) % 3][(j + 2) % 3] * T[(i + 2) % 3][(j + 1) % 3]) ** 2 for i in range(3) for j in range(3))
        return I1 * K / (9 * t * t) - 1
    raise ValueError(metric)


class _Plain:
    """The objective in plain torch, 64 bits."""

    def __init__(self, c):
        self.c, self.en = c, _elem_nodes(c)
        self.B, self.G, w = _rules(c)
        ww = w
        for _ in range(c["dim"] - 1):
            ww = (ww[:, None] * w[None, :]).reshape(-1)
        self.w = ww[None, :]
        if c["target"] == "local":
            det = _det(_jacobians(c, _positions(dict(c, jitter=0.0), 0)[0], self.en, self.B, self.G))
            self.s, self.detW = det ** (1.0 / c["dim"]), det
        else:
            self.s = _scale(c) if c["target"] == "scaled" else 1.0
            self.detW = self.s ** c["dim"]

    def F(self, x):
        A = _jacobians(self.c, x, self.en, self.B, self.G)
        T = [[t / self.s for t in row] for row in A]
        return (self.w * self.detW * _mu(self.c["metric"], T)).sum(), _det(A).min()

    def grad(self, x, fixed, graph=False):
        x = x.detach().requires_grad_(True)
        F, md = self.F(x)
        g, = torch.autograd.grad(F, x, create_graph=graph)
        return x, F.detach(), md.detach(), g * (~fixed)

    def hess(self, x, fixed):
        """v -> H(x) v on the free unknowns."""
        x, _, _, g = self.grad(x, fixed, graph=True)
        return lambda v: torch.autograd.grad((g * (v * (~fixed))).sum(), x, retain_graph=True)[0] * (~fixed)


def _minres(H, b, iters):
    """`iters` iterations of MINRES on H p = b from zero."""
    x, v_old, v = torch.zeros_like(b), torch.zeros_like(b), b.clone()
    beta = v.norm()
    v, eta = v / beta, beta
    g0 = g1 = 1.0
    s0 = s1 = 0.0
    w_old, w = torch.zeros_like(b), torch.zeros_like(b)
    beta = 0.0
    for _ in range(iters):
        u = H(v)
        a = (v * u).sum()
        u = u - a * v - beta * v_old
        beta_new = u.norm()
        d = g1 * a - g0 * s1 * beta
        r1, r2, r3 = torch.sqrt(d * d + beta_new * beta_new), s1 * a + g0 * g1 * beta, s0 * beta
        g0, s0, g1, s1 = g1, s1, d / r1, beta_new / r1
        w_old, w = w, (v - r3 * w_old - r2 * w) / r1
        x = x + g1 * eta * w
        eta = -s1 * eta
        v_old, v, beta = v, u / beta_new, beta_new
    return x


def _layers(net):
    dev = dict(device="cuda", dtype=torch.float64)
    p = [torch.tensor(a, **dev) for a in net.unflatten(net.get(0))]
    return [t.to(torch.bfloat16).double() if t.ndim == 2 else t for t in p]


def _forward(p, X):
    a1 = torch.relu(X @ p[0].T + p[1])
    a2 = torch.relu(a1 @ p[2].T + p[3])
    return a2 @ p[4].T + p[5]


def _patches(c, x):
    """Patch features [nelem][2 (3k+1)^2] of a 2D grid, before their rounding."""
    k, nx, ny = c["order"], c["nx"], c["ny"]
    p = x.reshape(2, k * ny + 1, k * nx + 1)

    def reflect(p, d):   # ghost nodes: point reflections through the boundary node of the same line
        lo = 2 * p.narrow(d, 0, 1) - p.narrow(d, 1, k).flip(d)
        m = p.shape[d]
        hi = 2 * p.narrow(d, m - 1, 1) - p.narrow(d, m - 1 - k, k).flip(d)
        return torch.cat([lo, p, hi], d)

    e = reflect(reflect(p, 2), 1)
    m = 3 * k + 1
    u = e.unfold(1, m, k).unfold(2, m, k)                       # [2, ny, nx, b, a]
    v = p[:, ::k, ::k]
    ctr = 0.25 * (v[:, :-1, :-1] + v[:, 1:, :-1] + v[:, :-1, 1:] + v[:, 1:, 1:])
    r = torch.tensor(mg.lattice_coordinates(k, 3) * 3 - 1.5, device="cuda")
    f = (u - ctr[..., None, None]) * nx
    f = torch.stack([f[0] - r[None, None, None, :], f[1] - r[None, None, :, None]], -1)
    return f.reshape(nx * ny, -1)


def exact(case, seed):
    c = dict(case)
    op = c["op"]
    if op == "mlp":
        st = prepare(case, seed)
        p = [t.requires_grad_(True) for t in _layers(st["net"])]
        X = st["X"].view(torch.bfloat16).double()[:, : st["net"].n_in]
        loss = ((_forward(p, X) - st["T"].double()) ** 2).sum() / c["batch"]
        g = torch.autograd.grad(loss, p)
        return {"loss": loss.detach(), "gradients": torch.cat([t.reshape(-1) for t in g])}
    x, fixed, gen = _positions(c, seed)
    if op == "newton":
        # with the unit square or cube's own uniform boundary, the uniform grid is the minimiser
        if c["deform"] == "shear":
            return None
        x, _ = _lattice(c)
        h = [1.0 / v for v in _sizes(c)]
        square = all(v == h[0] for v in h)
        return {"x": x if square else None, "min_det": float(np.prod(h)) if square else None, "status": 0}
    P = _Plain(c)
    if op == "step":
        v = torch.randn(x.shape, dtype=torch.float64, device="cuda", generator=gen)
        g = P.grad(x, fixed)[3]
        return [g, P.hess(x, fixed)(v)]
    if op == "hess":
        return P.hess(x, fixed)(torch.randn(x.shape, dtype=torch.float64, device="cuda", generator=gen))
    if op == "products":
        vs = [torch.randn(x.shape, dtype=torch.float64, device="cuda", generator=gen) for _ in range(c["count"])]
        H = P.hess(x, fixed)
        return [H(v) for v in vs]
    if op == "krylov":
        return _minres(P.hess(x, fixed), P.grad(x, fixed)[3], c["iters"])
    if op in ("trial", "autograd"):
        _, F, md, g = P.grad(x, fixed)
        return {"g": g, "F": F, "min_det": md} if op == "trial" else {"F": F, "g": g}
    st = prepare(case, seed)
    k, nx, ny = c["order"], c["nx"], c["ny"]
    Y = _forward(_layers(st["net"]), _patches(c, x).to(torch.bfloat16).double())
    xp = x.clone()
    own = Y.reshape(ny, nx, k, k, 2).permute(4, 0, 2, 1, 3).reshape(2, k * ny, k * nx) / nx
    xp.reshape(2, k * ny + 1, k * nx + 1)[:, :-1, :-1] += own * (~fixed).reshape(2, k * ny + 1, k * nx + 1)[:, :-1, :-1]
    F, md = P.F(xp)
    # the objective is compared where the displaced mesh is a valid one
    ok = bool(md > 0)
    return {"features": None, "x": xp, "F": F if ok else None, "min_det": md if ok else None, "Y": Y, "status": None}
