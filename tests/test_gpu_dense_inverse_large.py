"""The dense inverse of large coarse levels: beyond the rows of the panel kernel
(n > 5120) columns are eliminated one by one, in place; below, the working
matrices of a large inverse are given back after the build."""
import pytest

from paper_1912_12453_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def run(dim, level, precision):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build, chns
    build.build()
    g = (0.0, -1.0, 0.0) if dim == 2 else (0.0, 0.0, -1.0)
    prm = W.Params(dim, 1e-3, 0.1, 10.0, 5.0, 10.0, 1.0, 0.3, 0.5, gravity=g)
    wl = W.Workload("t", W.uniform_leaves(dim, level), prm, [W.Sphere((0.45, 0.5, 0.55)[:dim], 0.25)], False)
    mesh = chns.Mesh(wl.leaves)
    U0 = torch.from_numpy(W.initial_state(mesh.coords, wl).reshape(-1)).cuda()
    chns.init_mu(mesh, prm, U0)
    out = torch.empty_like(U0)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    st = chns.step(mesh, prm, U0, out, chns.SolverOpts.make(
        precision=precision, newton_rtol=1e-10, newton_atol=1e-16, krylov_rtol=1e-6, newton_max_it=12,
        reuse_preconditioner=0, preconditioner="multigrid", mg_coarsest=level))
    used = free - torch.cuda.mem_get_info()[0]
    F = chns.residual(mesh, prm, out, U0)
    F0 = chns.residual(mesh, prm, U0, U0)
    assert float(F.norm()) <= 1e-10 * float(F0.norm()) + 1e-16
    mesh.close()
    return st, used


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_columns_beyond_the_panel_rows(precision):
    st, _ = run(2, 5, precision)  # n = 5445
    # as for the smaller matrices: an inverse off by cond(J) eps along the weakest
    # directions; FP32 costs one more iteration for each of a few of them
    assert st["krylov_its_total"] <= (2 if precision == "fp64" else 10) * st["newton_its"]


@pytest.mark.parametrize("precision,size", [("fp64", 8), ("fp32", 4)])
def test_working_matrices_are_given_back(precision, size):
    n = 4374
    _, used = run(3, 3, precision)
    # kept: the inverse in double and in float, probing vectors and their slots in
    # 64 MB, vectors of n in a few MB; the two working matrices are not
    kept = n * n * (8 + 4)
    assert used <= kept + (64 << 20) + (24 << 20) < kept + 2 * n * n * size
