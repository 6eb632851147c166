"""FP32 J.w: no row is shifted as a whole by the rounding of its constants.

The roundings of values average out over the rows; what is left of
<y32 - y64, y64> / <y64, y64> is the error of the constants on the way of the row's
largest terms.  It stays within the last rounding, 2^-24, for phi and mu, and
within those of the increment's constant and of rho for the momentum."""
import pytest

from paper_1912_12453_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("schedule", [0, 5])
@pytest.mark.parametrize("dim,base,top,amp,dt", [(2, 5, 5, 0.02, 1e-3), (2, 5, 5, 0.5, 1e-1), (2, 4, 8, 0.02, 1e-3),
                                                 (3, 4, 4, 0.02, 5e-4), (3, 4, 4, 0.5, 1e-1), (3, 4, 6, 0.02, 5e-4),
                                                 (3, 6, 6, 0.02, 5e-4)])
def test_rows_are_not_shifted(dim, base, top, amp, dt, schedule):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1912_12453_gb300 import build, chns
    build.build()
    g = (0.0, -1.0, 0.0) if dim == 2 else (0.0, 0.0, -1.0)
    prm = W.Params(dim, dt, 0.04, 35.0, 125.0, 25.0, 1.0, 0.1, 0.1, gravity=g)
    sph = [W.Sphere((0.5, 0.45, 0.4)[:dim], 0.17)]
    leaves = W.uniform_leaves(dim, top) if base == top else W.band_leaves(dim, base, top, sph, 0.02)
    mesh = chns.Mesh(leaves)
    mesh.jacvec_schedule(schedule)
    U = torch.from_numpy(W.initial_state(mesh.coords, W.Workload("t", leaves, prm, sph, False)).reshape(-1)).cuda()
    n, nf = U.numel(), dim + 3
    gen = torch.Generator().manual_seed(n)

    def rand():
        return (2 * torch.rand(n, generator=gen, dtype=torch.float64) - 1).cuda()

    ut, dl = (0.95 * U + amp * rand()).float().double(), (0.01 * rand()).float().double()  # |phi| < 1 or no matter
    w = rand().float()
    new, old = ut + 0.5 * dl, ut - 0.5 * dl
    y = chns.jacvec(mesh, prm, new, old, w, precision="fp32").double().view(-1, nf)
    z = chns.jacvec(mesh, prm, new, old, w.double()).view(-1, nf)
    free = (y != w.double().view(-1, nf)).all(1)  # the constrained rows are w itself
    shift = ((y - z)[free] * z[free]).sum(0) / (z[free] ** 2).sum(0)
    for k in list(range(dim)) + [dim + 1, dim + 2]:
        assert abs(float(shift[k])) <= (2.0 ** -23 if k < dim else 2.0 ** -24), (k, float(shift[k]))
    mesh.close()
