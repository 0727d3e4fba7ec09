"""The one-cluster MINRES step writes its partial sums into the other blocks'
shared memory, which is allowed only once those blocks have begun to run."""
import os
import re

import numpy as np
import pytest

from paper_1807_09807_gb300 import meshgen as mg

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1807_09807_gb300", "csrc")


def test_cluster_barrier_before_the_first_remote_store():
    """In every kernel that works as a cluster: arrive on entry, and wait at
    the place the first reduction gives for it, which lies before its store."""
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "tmop_vec.cu")).read())
    reduce = src[src.index("double cluster_sum("):]
    assert reduce.index("before();") < reduce.index("map_shared_rank")
    kernels = [k for k in re.split(r"__global__", src)[1:] if "this_cluster()" in k]
    assert kernels
    for k in kernels:
        calls = re.findall(r"cluster_sum<NT>\([^;]*;", k)
        assert k.index("barrier_arrive()") < k.index("cluster_sum<NT>(")
        assert "barrier_wait()" in calls[0] and all("barrier_wait" not in c for c in calls[1:])


@pytest.mark.gpu
@pytest.mark.parametrize("nx", [(2, 2), (16, 16), (31, 31), (40, 40)])   # both block sizes
def test_blocks_that_start_late(nx):
    """Solves beside kernels that fill the GPU, so that a cluster's blocks wait
    for room: the same digits as on an idle GPU (deterministic sums)."""
    import torch
    from paper_1807_09807_gb300 import tmop as tm

    def mesh(n):
        x, en, fx = mg.structured(2, 1, n)
        x = np.ascontiguousarray(mg.jitter(x, fx, 0.1 / max(n), 5))
        return mg.Mesh(dim=2, order=1, nx=n, x=x, x_ideal=x, elem_nodes=en, fixed=fx, nq=3, quad_kind=mg.GL, metric=2)

    m, big = mesh(nx), mesh((400, 400))
    ctx, load = tm.Context.from_mesh(m), tm.Context.from_mesh(big)
    ctx.set_deterministic(True)
    x, xb = torch.tensor(m.x, device="cuda"), torch.tensor(big.x, device="cuda")
    b = torch.tensor(np.random.default_rng(3).standard_normal(m.x.shape) * (1 - m.fixed), device="cuda")
    p, it = ctx.krylov_solve(x, b, krylov_rtol=1e-10, krylov_maxit=60)
    p = p.clone()
    torch.cuda.synchronize()
    other = torch.cuda.Stream()
    for _ in range(8):
        with torch.cuda.stream(other):
            for _ in range(40):
                load.gradient(xb)
        q, jt = ctx.krylov_solve(x, b, krylov_rtol=1e-10, krylov_maxit=60)
        assert jt == it and torch.equal(q, p)
    torch.cuda.synchronize()
