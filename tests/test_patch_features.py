"""Patch features of every order, at the grid's edges (ghost nodes) and inside
it, against the definition evaluated in numpy with the same operations in
FP64; the fused multiply-subtract of the kernel may round the value before the
conversion to bfloat16 differently, which moves a feature by at most one
bfloat16 step, and only where it lies on a rounding boundary."""
import numpy as np
import pytest

from paper_1807_09807_gb300 import meshgen as mg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,nx", [(1, (1, 1)), (1, (5, 3)), (2, (3, 4)), (3, (6, 5)), (4, (4, 3))])
def test_patch_features_match_their_definition(order, nx):
    import torch
    from paper_1807_09807_gb300 import learned as L
    k = order
    x, en, fx = mg.structured(2, k, nx)
    x = mg.jitter(x, np.zeros_like(fx), 0.1 / (k * max(nx)), 7)
    m = mg.Mesh(dim=2, order=k, nx=nx, x=x, x_ideal=x, elem_nodes=en, fixed=fx)
    ldf = (L.n_features(k) + 7) // 8 * 8
    got = L.features(m, torch.tensor(x, device="cuda"), ldf).cpu().view(torch.bfloat16).double().numpy()
    p = x.reshape(2, k * nx[1] + 1, k * nx[0] + 1)

    def ghost(p, axis):   # point reflections through the boundary node of the same grid line
        p = np.moveaxis(p, axis, 0)
        n = p.shape[0]
        lo = [2 * p[0] - p[i] for i in range(k, 0, -1)]
        hi = [2 * p[-1] - p[n - 1 - i] for i in range(1, k + 1)]
        return np.moveaxis(np.concatenate([lo, p, hi]), 0, axis)

    e = ghost(ghost(p, 2), 1)
    side = 3 * k + 1
    ref = mg.lattice_coordinates(k, 3) * 3 - 1.5
    for ey in range(nx[1]):
        for ex in range(nx[0]):
            c = 0.25 * (p[:, k * ey, k * ex] + p[:, k * ey, k * ex + k] + p[:, k * ey + k, k * ex] +
                        p[:, k * ey + k, k * ex + k])
            u = (e[:, k * ey:k * ey + side, k * ex:k * ex + side] - c[:, None, None]) * nx[0]
            f = np.stack([u[0] - ref[None, :], u[1] - ref[:, None]], -1).reshape(-1)
            row = got[ex + nx[0] * ey]
            assert np.all(np.abs(row[:f.size] - f) <= 2.0 ** -8 * np.abs(f) + 1e-13), (ex, ey)
            assert not row[f.size:].any()
