"""FP32 J.w of small uniform meshes, straight from the states (65,536 corners at
most: level 7 in 2D, level 4 in 3D; one level more takes the prepared path)."""
import pytest

from paper_1912_12453_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,level", [(2, 1), (2, 3), (2, 7), (2, 8), (3, 1), (3, 2), (3, 4), (3, 5)])
def test_states_path(dim, level):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build, chns
    build.build()
    g = (0.0, -1.0, 0.0) if dim == 2 else (0.0, 0.0, -1.0)
    prm = W.Params(dim, 1e-3, 0.1, 10.0, 5.0, 10.0, 1.0, 0.3, 0.5, gravity=g)
    mesh = chns.Mesh(W.uniform_leaves(dim, level))
    n = mesh.coords.shape[0] * (dim + 3)
    gen = torch.Generator().manual_seed(level)
    old = (0.8 * (2 * torch.rand(n, generator=gen, dtype=torch.float64) - 1)).cuda()  # |phi| < 1: no clip to flip
    new = (old.cpu() + 0.1 * torch.rand(n, generator=gen, dtype=torch.float64)).cuda()
    w = (2 * torch.rand(n, generator=gen) - 1).cuda()
    y = chns.jacvec(mesh, prm, new, old, w, precision="fp32")
    # about 60 roundings of 6e-8 a term, terms that cancel by up to four
    y64 = chns.jacvec(mesh, prm, new, old, w.double())
    assert float((y.double() - y64).norm()) <= 1.5e-5 * float(y64.norm())
    if dim == 3:  # states on 8-byte boundaries take the prepared path: the same bits
        odd = torch.empty(n + 1, device="cuda", dtype=torch.float64)[1:]
        odd.copy_(new)
        assert torch.equal(chns.jacvec(mesh, prm, odd, old, w, precision="fp32"), y)
    mesh.close()
