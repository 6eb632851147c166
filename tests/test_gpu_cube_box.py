"""FP64 residual and J.w on a box with equal sides (in 3D: constants per leaf,
plain differences) against the general form, which a box a few last bits off
takes."""
import pytest

from paper_1912_12453_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("side", [1.0, 0.7, 3.0])
@pytest.mark.parametrize("dim,base,top", [(2, 1, 1), (2, 2, 5), (3, 1, 1), (3, 2, 4)])
@pytest.mark.parametrize("eta,rho", [(0.5, 0.3), (1.0, 1.0)])  # 1: eta' and rho' are 0, one of them -0
def test_cube_matches_general_form(dim, base, top, side, eta, rho):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build, chns
    build.build()
    g = (0.3, -1.0, 0.0) if dim == 2 else (0.3, -0.2, -1.0)
    prm = W.Params(dim, 1e-3, 0.1, 10.0, 5.0, 10.0, 1.0, rho, eta, gravity=g)
    leaves = W.uniform_leaves(dim, top) if base == top else W.band_leaves(
        dim, base, top, [W.Sphere((0.45, 0.5, 0.55)[:dim], 0.25)], 0.05)
    off = side * (1.0 + 2.0 ** -50)
    boxes = [(side, side, side), (side, off, side)]
    meshes = [chns.Mesh(leaves, lo=(0.0, 0.0, 0.0), hi=b) for b in boxes]
    n = meshes[0].n_dof
    gen = torch.Generator().manual_seed(dim * 10 + top)
    old = (0.8 * (2 * torch.rand(n, generator=gen, dtype=torch.float64) - 1)).cuda()  # |phi| < 1: no clip to flip
    new = old + (0.1 * torch.rand(n, generator=gen, dtype=torch.float64)).cuda()
    w = (2 * torch.rand(n, generator=gen, dtype=torch.float64) - 1).cuda()
    f = (2 * torch.rand(n, generator=gen, dtype=torch.float64) - 1).cuda()
    nf = dim + 3
    for call in (lambda m: chns.residual(m, prm, new, old), lambda m: chns.residual(m, prm, new, old, forcing=f),
                 lambda m: chns.jacvec(m, prm, new, old, w)):
        a, b = (call(m).view(-1, nf) for m in meshes)
        # the boxes differ by 1e-15, a term by at most 8 powers of a side, and each
        # form rounds a term about 60 times at 1e-16; row by row of the fields
        for k in range(nf):
            assert float((a[:, k] - b[:, k]).norm()) <= 1e-13 * float(b[:, k].norm()) + 1e-300
    for m in meshes:
        m.close()
