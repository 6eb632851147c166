"""FP64 in 3D: the mass term of the phi row is not shifted by the rounding of the
constants.

With v = 0 and mu = 0 the row is M d / dt, in the residual (d the increment) as in
J.w (d the direction).  The shift of a row is <y - z, z> / <z, z> against z in
extended precision: the roundings of values average out over the nodes, that of
1/dt (up to 2^-53) over sixteen time steps.  What is left is the constants' share,
within half a rounding, 2^-54."""
import numpy as np
import pytest

from paper_1912_12453_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["residual", "jacvec"])
@pytest.mark.parametrize("hi", [(1.0, 1.0, 1.0), (1.0, 1.0, 2.0)], ids=["cube", "box"])
def test_mass_term(call, hi):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    if np.finfo(np.longdouble).nmant <= 52:
        pytest.skip("no extended precision")
    from paper_1912_12453_gb300 import build, chns
    build.build()
    level = 4
    mesh = chns.Mesh(W.uniform_leaves(3, level), hi=hi)
    n1 = (1 << level) + 1
    at = mesh.coords_int @ np.array([1, n1, n1 * n1])  # node -> place in the grid
    L = np.longdouble
    # 1D mass matrix of the n1 nodes, in units of h / 6
    m = 4 * np.eye(n1) + np.eye(n1, k=1) + np.eye(n1, k=-1)
    m[0, 0] = m[-1, -1] = 2
    m = m.astype(L)
    h3 = L(hi[0]) * L(hi[1]) * L(hi[2]) / 8 ** level / 216
    rng = np.random.default_rng(3)
    shifts = []
    for dt in 10.0 ** rng.uniform(-3.6, -3.0, 16):
        prm = W.Params(3, float(dt), 0.1, 10.0, 5.0, 10.0, 1.0, 0.3, 0.5)
        d = rng.uniform(-1.0, 1.0, mesh.n_nodes)
        grid = np.zeros(n1 ** 3, dtype=L)
        grid[at] = d.astype(L)
        z = np.einsum("ai,bj,ck,ijk->abc", m, m, m, grid.reshape(n1, n1, n1), optimize=True).reshape(-1)[at] * h3 / L(dt)
        u = np.zeros((mesh.n_nodes, 6))
        u[:, 4] = d
        u, zero = torch.from_numpy(u.reshape(-1)).cuda(), torch.zeros(mesh.n_dof, dtype=torch.float64, device="cuda")
        if call == "residual":
            y = chns.residual(mesh, prm, u, zero)
        else:
            y = chns.jacvec(mesh, prm, zero, zero, u)
        y = y.view(-1, 6)[:, 4].cpu().numpy().astype(L)
        shifts.append(float(((y - z) * z).sum() / (z * z).sum()))
    assert abs(np.mean(shifts)) <= 2.0 ** -54, np.mean(shifts)
    mesh.close()
