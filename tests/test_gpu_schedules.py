"""A fixed FP32 J.w schedule is the one that runs, on small meshes too, and the
schedules with two Gauss points per lane differ in their launch shape only."""
import pytest

from paper_1912_12453_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def setup(leaves):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build, chns
    build.build()
    dim = leaves.dim
    g = (0.0, -1.0, 0.0) if dim == 2 else (0.0, 0.0, -1.0)
    prm = W.Params(dim, 1e-3, 0.1, 10.0, 5.0, 10.0, 1.0, 0.3, 0.5, gravity=g)
    mesh = chns.Mesh(leaves)
    n = mesh.coords.shape[0] * (dim + 3)
    gen = torch.Generator().manual_seed(n)
    old = 0.8 * (2 * torch.rand(n, generator=gen, dtype=torch.float64) - 1)
    new = old + 0.1 * torch.rand(n, generator=gen, dtype=torch.float64)
    w = 2 * torch.rand(n, generator=gen) - 1
    new, old, w = new.cuda(), old.cuda(), w.cuda()
    return torch, chns, mesh, lambda: chns.jacvec(mesh, prm, new, old, w, precision="fp32")


@pytest.mark.parametrize("dim,level", [(2, 3), (2, 7), (3, 2), (3, 4)])
def test_a_fixed_schedule_runs_on_a_small_mesh(dim, level):
    torch, chns, mesh, apply = setup(W.uniform_leaves(dim, level))

    def launches():
        n = chns.kernel_launches()
        y = apply()
        return chns.kernel_launches() - n, y

    n0, y0 = launches()
    assert n0 == 2  # straight from the states: element kernel and node gather
    for v in (0, 1, 2, 3):
        mesh.jacvec_schedule(v)
        n, y = launches()
        assert n == 3  # preparation, the schedule's element kernel, node gather
        assert torch.equal(y, y0)
    mesh.close()


@pytest.mark.parametrize("leaves", ["uniform", "band"])
def test_two_point_schedules_agree_on_large_meshes(leaves):
    leaves = W.uniform_leaves(3, 6) if leaves == "uniform" else W.band_leaves(
        3, 4, 7, [W.Sphere((0.45, 0.5, 0.55), 0.25)], 0.04)
    torch, chns, mesh, apply = setup(leaves)
    y0 = apply()
    for v in (1, 2, 3):
        mesh.jacvec_schedule(v)
        assert torch.equal(apply(), y0)
    mesh.close()
