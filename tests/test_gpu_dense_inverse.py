"""The dense inverse of the coarsest level (blocked Gauss-Jordan).

On a uniform mesh that is its own coarsest multigrid level the preconditioner
is the inverse of the whole Jacobian.  Built anew for each Newton iteration, it
leaves FGMRES a couple of iterations, whatever the panel width, the rows per
thread and the remainder of the last panel (matrix sizes 45 to 4374).
"""
import pytest

from paper_1912_12453_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("dim,level", [(2, 1), (2, 2), (2, 3), (2, 4), (3, 1), (3, 2), (3, 3)])
def test_exact_bottom_solve(dim, level, precision):
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
    st = chns.step(mesh, prm, U0, out, chns.SolverOpts.make(
        precision=precision, newton_rtol=1e-10, newton_atol=1e-16, krylov_rtol=1e-6, newton_max_it=12,
        reuse_preconditioner=0, preconditioner="multigrid", mg_coarsest=level))
    # FP64: the inverse is off by cond(J) eps <= 1e9 x 1e-16 along the weakest
    # direction, so one iteration gains 1e-7 and two are enough for 1e-6.
    # FP32: off by O(1) along a few pressure directions only, each of which
    # costs one more iteration.
    assert st["krylov_its_total"] <= (2 if precision == "fp64" else 10) * st["newton_its"]
    F = chns.residual(mesh, prm, out, U0)
    F0 = chns.residual(mesh, prm, U0, U0)
    assert float(F.norm()) <= 1e-10 * float(F0.norm()) + 1e-16
    mesh.close()
