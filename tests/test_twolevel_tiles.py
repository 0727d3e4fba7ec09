"""The sine transforms of the two-level preconditioner at the edges of their
tiles (8 outputs per side, 32-deep chunks): 16, 17, 33 and 65 interior
vertices along an axis, against the dense definition in oracle/twolevel.py
(1e-10: FP64 sums of at most 65 terms, times the condition number ~1e3 of the
coarse Laplacian)."""
import numpy as np
import pytest

import oracle
from paper_1807_09807_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,order,nx", [(2, 1, (17, 18)), (2, 2, (34, 17)), (2, 1, (66, 18)), (3, 1, (18, 3, 4))])
def test_coarse_part_at_tile_edges(dim, order, nx):
    import torch
    from oracle import twolevel as otl
    from paper_1807_09807_gb300 import tmop as tm
    x, en, fx = mg.structured(dim, order, nx)
    x = mg.jitter(x, fx, 0.05 / (order * max(nx)), 3)
    m = mg.Mesh(dim=dim, order=order, nx=nx, x=x, x_ideal=x, elem_nodes=en, fixed=fx, nq=order + 1,
                metric=2 if dim == 2 else 303)
    ctx = tm.Context.from_mesh(m)
    orc = oracle.Problem(m.dim, m.order, m.elem_nodes, m.nnode, m.fixed, m.nq, m.metric)
    r = np.random.default_rng(4).standard_normal(x.shape) * (1 - fx)
    xd, rd = torch.tensor(x, device="cuda"), torch.tensor(r, device="cuda")
    z2, a = ctx.precond_apply(xd, rd, 2)
    z1, _ = ctx.precond_apply(xd, rd, 1)
    ref_a = otl.alpha(lambda v: orc.hess_apply(x, v), nx, order, dim)
    assert abs(a - ref_a) <= 1e-10 * ref_a
    ref = otl.coarse_part(r, nx, order, ref_a)
    assert np.linalg.norm((z2 - z1).cpu().numpy() - ref) <= 1e-10 * np.linalg.norm(ref)
