"""States that start on an 8-byte boundary only: the 3D residual kernel reads
pairs, so such views go through a copy and give the same numbers."""
import pytest

from paper_1912_12453_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("odd", [(1, 0), (0, 1), (1, 1)])
def test_odd_views(dim, odd):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build, chns
    build.build()
    g = (0.0, -1.0, 0.0) if dim == 2 else (0.0, 0.0, -1.0)
    prm = W.Params(dim, 1e-3, 0.1, 10.0, 5.0, 10.0, 1.0, 0.3, 0.5, gravity=g)
    sph = [W.Sphere((0.45, 0.5, 0.55)[:dim], 0.25)]
    wl = W.Workload("t", W.band_leaves(dim, 2, 4, sph, 0.05), prm, sph, False)
    mesh = chns.Mesh(wl.leaves)
    old = torch.from_numpy(W.initial_state(mesh.coords, wl).reshape(-1)).cuda()
    new = old + 1e-2 * torch.sin(torch.arange(old.numel(), device="cuda", dtype=torch.float64))
    views = []
    for U, o in zip((new, old), odd):
        b = torch.empty(U.numel() + 1, device="cuda", dtype=torch.float64)
        v = b[o:o + U.numel()]
        v.copy_(U)
        assert v.data_ptr() % 16 == 8 * o
        views.append(v)
    for prec in ("fp64", "fp32"):
        w = torch.cos(torch.arange(old.numel(), device="cuda", dtype=torch.float64)).to(
            torch.float64 if prec == "fp64" else torch.float32)
        assert torch.equal(chns.jacvec(mesh, prm, *views, w, precision=prec),
                           chns.jacvec(mesh, prm, new, old, w, precision=prec))
    assert torch.equal(chns.residual(mesh, prm, *views), chns.residual(mesh, prm, new, old))
    assert chns.tau_floor_count(mesh, prm, *views) == chns.tau_floor_count(mesh, prm, new, old)
    mesh.close()
