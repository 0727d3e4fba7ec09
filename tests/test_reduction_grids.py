"""MINRES reductions on both sides of the sizes at which their grid changes:
one value per thread up to 304 blocks of 256, then up to four values, then more
blocks. After twelve iterations the oracle's iterate (1e-10, the FP32 form's
operator and vectors 1e-4)."""
import numpy as np
import pytest

import oracle
from paper_1807_09807_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,unknowns", [((151, 255), 77824), ((150, 257), 77916), ((303, 511), 311296), ((302, 514), 312090)])
@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_minres_at_the_edges_of_the_grids(nx, unknowns, precision):
    import torch
    from paper_1807_09807_gb300 import tmop as tm
    x, en, fx = mg.structured(2, 1, nx)
    x = np.ascontiguousarray(mg.jitter(x, fx, 0.08 / max(nx), 5))
    assert x.size == unknowns
    m = mg.Mesh(dim=2, order=1, nx=nx, x=x, x_ideal=x, elem_nodes=en, fixed=fx, nq=2, quad_kind=mg.GL, metric=2)
    orc = oracle.Problem(2, 1, en, m.nnode, fx, 2, 2)
    ctx = tm.Context.from_mesh(m, precision=tm.FP64 if precision == "fp64" else tm.FP32_MIXED)
    xd = torch.tensor(x, device="cuda")
    b = np.random.default_rng(3).standard_normal(x.shape) * (1 - fx)
    bd = torch.tensor(b, device="cuda")
    p, _ = ctx.krylov_solve(xd, bd, krylov_rtol=1e-14, krylov_maxit=12)
    po, _ = orc.minres(x, b, rtol=1e-14, maxit=12)
    assert np.linalg.norm(p.cpu().numpy() - po) <= (1e-10 if precision == "fp64" else 1e-4) * np.linalg.norm(po)
